"""Uploads at the memory budget's limits: what is refused leaves nothing behind."""

import numpy as np
import pytest

from synth import Scene

pytestmark = pytest.mark.gpu


def _scene(n):
    rng = np.random.default_rng(n)
    c = rng.uniform((-1.5, -1, 2), (1.5, 1, 6), (n, 1, 3))
    v = (c + 0.05 * rng.uniform(-1, 1, (n, 3, 3))).astype(np.float32).reshape(-1, 3)
    return Scene(v, np.arange(3 * n, dtype=np.uint32).reshape(n, 3), np.zeros(n, np.uint32), 1)


def test_a_budget_without_room_for_the_wide_tree_leaves_no_error_behind():
    """The budget admits the triangles and the binary tree but not the 4-wide nodes: the upload
    reports that, gives back what it took and leaves no error pending for the next library's check on
    this thread."""
    import torch
    from paper_2210_06158_gb300 import dof
    n = 5000
    with_all = dof.Context(0)
    sc = dof.Scene(with_all, _scene(n))
    total = with_all.bytes_in_use
    assert sc.info().n_nodes4 > 100
    ctx = dof.Context(0, mem_budget_bytes=total - 1024)
    with pytest.raises(dof.DofError) as e:
        dof.Scene(ctx, _scene(n))
    assert e.value.code == -3
    assert ctx.bytes_in_use == 0
    x = torch.ones(1000, device="cuda") * 2         # a launch whose error check is torch's
    torch.cuda.synchronize()
    assert float(x.sum()) == 2000.0


@pytest.mark.parametrize("n", [1, 2, 37, 5001])
def test_a_scene_takes_what_its_parts_take(n):
    """48 bytes per triangle and 4 for its index, 64 per binary node, 128 per 4-wide node, nothing for
    padding: a budget of just that admits it, a byte less does not."""
    from paper_2210_06158_gb300 import dof
    ctx = dof.Context(0)
    i = dof.Scene(ctx, _scene(n)).info()
    total = 52 * n + 64 * (n - 1) + 128 * i.n_nodes4
    assert i.device_bytes == total
    exact = dof.Context(0, mem_budget_bytes=total)
    sc = dof.Scene(exact, _scene(n))
    assert exact.bytes_in_use == total
    sc.close()
    assert exact.bytes_in_use == 0
    with pytest.raises(dof.DofError) as e:
        dof.Scene(dof.Context(0, mem_budget_bytes=total - 1), _scene(n))
    assert e.value.code == -3


def test_kept_scratch_stays_within_what_the_budget_leaves():
    """The upload's scratch (over 300 MB here) is kept for the next one only as far as the budget has
    room beside the scene, and a history that takes the room takes it from the kept scratch."""
    import torch
    from paper_2210_06158_gb300 import dof
    host = _scene(1_000_000)
    first = dof.Context(0)
    sc = dof.Scene(first, host)
    total = first.bytes_in_use
    sc.close()
    first.close()
    room = 32 << 20
    ctx = dof.Context(0, mem_budget_bytes=total + room)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]

    def kept():
        torch.cuda.synchronize()
        return free - torch.cuda.mem_get_info()[0] - ctx.bytes_in_use

    sc = dof.Scene(ctx, host)
    assert kept() <= room + (8 << 20)                  # the allocator rounds up to pages of 2 MB
    hist = dof.History(ctx, 640, 360)
    # the history's some forty buffers are each rounded up to pages
    assert kept() <= total + room - ctx.bytes_in_use + (88 << 20)
    hist.close()
    sc.close()
    assert ctx.bytes_in_use == 0
