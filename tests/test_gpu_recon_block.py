"""The reconstruction's block is the caller's in a step that holds small sessions too, and no
instance of it keeps registers in memory."""

import re
from pathlib import Path

import pytest

from synth import make_workload


@pytest.mark.gpu
def test_the_block_of_large_sessions_stands_beside_a_small_one():
    """A graph captured with one block refuses to replay with another, small session or not."""
    import torch
    from paper_2210_06158_gb300 import dof
    ctx = dof.Context(0)
    items = []
    for k, (W, H) in enumerate([(130, 74), (642, 362)]):
        w = make_workload("c1", W=W, H=H, session=k)
        sc = dof.Scene(ctx, w.scene)
        gb = dof.gbuffer(ctx, sc, w.camera(0), w.params, W, H)
        items.append(dict(scene=sc, gbuf=gb, cam=w.camera(0), params=dict(w.params), hist=dof.History(ctx, W, H, max_rays=1)))
    ctx.set_gather(recon_block=(16, 16))
    g = dof.Graph(ctx, items)
    g.launch(items)
    torch.cuda.synchronize()
    ctx.set_gather(recon_block=(32, 8))
    with pytest.raises(dof.DofError) as e:
        g.launch(items)
    assert e.value.code == -7
    g.close()


def test_no_instance_of_the_reconstruction_spills():
    log = Path(__file__).resolve().parents[1] / "paper_2210_06158_gb300" / "_lib" / "obj" / "recon.ptxas.txt"
    if not log.exists():
        pytest.skip("the library has not been built here")
    found = re.findall(r"Compiling entry function '(\S*k_recon\S*)'.*?(\d+) bytes spill stores, (\d+) bytes spill loads",
                       log.read_text(), re.S)
    assert len(found) >= 6
    # the instance for mixed image storage holds both storages' taps and may keep a few words in memory
    bad = [f for f in found if (int(f[1]) or int(f[2])) and "Li2E" not in f[0]]
    assert not bad, bad
