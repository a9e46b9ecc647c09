"""The autotuner's choices on a stand-in context (host only): the cache key
tells operators and sets of forms apart, a cached choice that the context refuses
is timed again, what lbm_create picks is tried whatever the context was set to,
and the box form is timed with the steps its graph needs."""
import json
import types

import pytest

torch = pytest.importorskip("torch")
from paper_1904_03618_gb300 import autotune, lbm  # noqa: E402


class Context:
    """A 40 x 30 x 20 MRT lattice: the box form fastest, then (8, 16, 2)."""

    def __init__(self, bgk=False):
        self.bgk, self.config, self.box, self.steps = bgk, (8, 4, 0), 0, []


def _set(ctx, ty, zc, hold):
    if ctx.bgk and (ty, hold) != (8, 2):
        raise lbm.LbmError(lbm.LBM_ERR_ARG, "refused")
    ctx.config, ctx.box, ctx.steps = (ty, zc, hold), 0, []


@pytest.fixture
def tuner(monkeypatch):
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda *a: "GPU")
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch.cuda, "get_device_properties",
                        lambda d: types.SimpleNamespace(multi_processor_count=152))
    monkeypatch.setattr(lbm, "lbm_set_fused_config", _set)
    monkeypatch.setattr(lbm, "lbm_get_fused_config", lambda c: c.config)
    monkeypatch.setattr(lbm, "lbm_set_box", lambda c, b: setattr(c, "box", b), raising=False)
    monkeypatch.setattr(lbm, "lbm_get_box", lambda c: c.box, raising=False)
    monkeypatch.setattr(lbm, "lbm_step", lambda c, n: c.steps.append(n))

    class Event:
        def __init__(self, **kw):
            pass

        def record(self, stream):
            pass

        def elapsed_time(self, other):
            c = tuner_ctx[0]
            return c.steps[-1] * (1.0 if c.box else 2.0 if c.config == (8, 16, 2) else 3.0)

    monkeypatch.setattr(torch.cuda, "Event", Event)
    tuner_ctx = [None]

    def tune(ctx, p, **kw):
        tuner_ctx[0] = ctx
        return autotune.tune(ctx, [p], types.SimpleNamespace(synchronize=lambda: None), **kw)
    return tune


def _p(**kw):
    return lbm.make_params(40, 30, 20, **kw)


def test_the_default_form_is_tried_and_timed_with_its_graph(tuner, tmp_path):
    cache = str(tmp_path / "t.json")
    ctx = Context()
    ty, zc, hold, ms, source = tuner(ctx, _p(), cache_path=cache)
    assert source == "timed" and ms == 1.0 and ctx.box == lbm.lbm_default_box(_p()) == 2
    assert (ty, zc, hold) == ctx.config == lbm.lbm_default_fused_config(_p(), 152)
    again = Context()
    assert tuner(again, _p(), cache_path=cache)[4] == "cache"
    assert again.box == 2 and again.config == ctx.config
    again.steps = []
    autotune._time(again, types.SimpleNamespace(synchronize=lambda: None), 8)
    assert again.steps == [20, 32]  # a graph of 16 steps captured, then replayed twice
    # configurations the caller names run without it
    ctx = Context()
    assert tuner(ctx, _p(), cache_path=None, candidates=[(8, 12, 2), (8, 16, 2)])[:3] == (8, 16, 2)
    assert ctx.box == 0


def test_operators_have_their_own_entries(tuner, tmp_path):
    cache = str(tmp_path / "t.json")
    tuner(Context(), _p(), cache_path=cache, candidates=[(15, 32, 7)])
    bgk = _p(collision="bgk")
    assert autotune.signature([bgk], 0) != autotune.signature([_p()], 0)
    ctx = Context(bgk=True)
    got = tuner(ctx, bgk, cache_path=cache)
    assert got[4] == "timed" and got[:3] == (8, 16, 2) and ctx.box == 0


def test_a_refused_or_older_entry_is_timed_again(tuner, tmp_path):
    cache = str(tmp_path / "t.json")
    bgk = _p(collision="bgk")
    key = autotune.signature([bgk], 0)
    for entry in (dict(tile_y=12, zchunk=6, hold=7, box=0, ms=1.0),
                  dict(tile_y=8, zchunk=12, hold=2, ms=1.0)):
        (tmp_path / "t.json").write_text(json.dumps({key: entry}))
        got = tuner(Context(bgk=True), bgk, cache_path=cache)
        assert got[4] == "timed" and got[:3] == (8, 16, 2)
