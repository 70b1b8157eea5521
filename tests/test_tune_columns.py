"""The gather tuner reaches the block that the library itself takes for the main filter's columns."""
import types

import pytest

from paper_2210_06158_gb300 import tune


def _run(monkeypatch, cost):
    import torch
    clock = [0.0]

    class Event:
        def __init__(self, enable_timing=True):
            self.t = None

        def record(self, stream=None):
            self.t = clock[0]

        def synchronize(self):
            pass

        def elapsed_time(self, end):
            return end.t - self.t

    monkeypatch.setattr(torch.cuda, "Event", Event)
    cfg, tried = dict(block=(32, 8), form=0), []        # as the warm-up frames find the context

    def set_gather(block, main_form, recon_block):
        cfg.update(block=tuple(block), form=main_form)
        tried.append((main_form, tuple(block)))

    def run_frame(k):
        clock[0] += cost(cfg["form"], cfg["block"])

    best, _ = tune.tune_gathers(types.SimpleNamespace(set_gather=set_gather), run_frame, frames=2,
                                stream=types.SimpleNamespace())
    return best, tried


def test_columns_end_with_their_own_block(monkeypatch):
    def cost(form, block):
        if form != 3:
            return 1.2
        return 1.0 if block == (32, 2) else 1.1

    best, _ = _run(monkeypatch, cost)
    assert best["main_form"] == 3 and best["gather_block"] == (32, 2)


@pytest.mark.parametrize("form", [0, 1, 2])
def test_the_other_forms_are_not_timed_with_it(monkeypatch, form):
    best, tried = _run(monkeypatch, lambda f, b: 1.0 if f == form else 1.2)
    assert best["main_form"] == form
    assert not [t for t in tried if t[1] == (32, 2)]
