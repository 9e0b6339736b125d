"""Which steps are recorded as graphs and replayed, and what the context keeps of them."""
import numpy as np
import pytest
import torch

from paper_2601_20332_b200 import binding as wd
from paper_2601_20332_b200 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"
BF16 = dict(dtype="bf16", dh=128, Hq=2, Hkv=2, F=704)       # the small model with the widths of the tensor-core path


def _context(name="tiny", **over):
    cfg = synth.get_config(name, P=20, G=140, **over)
    ids = synth.make_prompts(cfg)
    S = ids.shape[1]
    return cfg, ids, wd.Context(cfg, synth.make_weights(cfg, DEV), 1, S, S, 128)


def _steps(st, windows, stream):
    """A step for each number of active positions, ten at a time behind one of 64, so that they find steps queued.  They unmask nothing
    (the same window can be taken again), and only the first step of a state refreshes."""
    for i in range(0, len(windows), 10):
        for A in [64] + windows[i:i + 10]:
            st.step(A, 128 - A, 1000, 1, 0, stream)
        st.sync_all()


def test_fp32_steps_synced_one_by_one():
    """With nothing queued an fp32 configuration is recorded after it has come 32 times.  A graph's kernels write the context's logits:
    the tap of a step is filled behind them, and left alone by the other steps."""
    runs = []
    for on in (False, True):
        cfg, ids, ctx = _context()
        ctx.set_graphs(on)
        stream = torch.cuda.Stream(device=DEV)
        st = wd.State(ctx, ids)
        taps = [torch.full((128, cfg["V"]), -1.0, device=DEV) for _ in range(2)]
        torch.cuda.synchronize()
        got, stats = [], []
        for i in range(1 + 48):                 # a refresh, then normal steps of one configuration
            st.set_taps(logits=taps[i % 3] if i % 3 < 2 else None)
            st.step(8, 120, 1000, 1, 1, stream)
            out = st.sync()
            got.append([t.clone() for t in taps] + [out["positions"], out["token_ids"], out["confidence"]])
            stats.append(ctx.graph_stats())
            for t in taps:
                t.fill_(-1.0)
            torch.cuda.synchronize()
        runs.append((got, stats))
        st.close()
        ctx.close()
    for i, (a, b) in enumerate(zip(runs[0][0], runs[1][0], strict=True)):
        for j in range(2):
            assert torch.equal(a[j], b[j])
            assert bool((b[j][:8] != -1.0).all()) == (i % 3 == j) and bool((b[j][8:] == -1.0).all())
        assert all(np.array_equal(x, y) for x, y in zip(a[2:], b[2:], strict=True))
    assert runs[0][1][-1] == (0, 0)
    assert runs[1][1][32:34] == [(0, 0), (1, 0)] and runs[1][1][-1] == (1, 15)


def test_graphs_of_destroyed_states_make_room():
    """A state that filled the context's graphs and is gone does not keep the next one's steps from being recorded."""
    cfg, ids, ctx = _context()
    stream = torch.cuda.Stream(device=DEV)
    st = wd.State(ctx, ids)
    _steps(st, list(range(1, 41)), stream)      # more windows than there is room for
    st.close()
    captured, replayed = ctx.graph_stats()
    assert captured == 32 and replayed == 0
    st = wd.State(ctx, ids)
    _steps(st, [8] * 10, stream)
    assert ctx.graph_stats() == (captured + 1, replayed + 9)
    st.close()
    ctx.close()


def test_a_window_that_keeps_coming_back_is_counted():
    """With nothing queued a bf16 configuration is recorded after it has come eight times, however many windows that come once lie
    between."""
    cfg, ids, ctx = _context(**BF16)
    stream = torch.cuda.Stream(device=DEV)
    st = wd.State(ctx, ids)

    def step(A):
        st.step(A, 128 - A, 1000, 1, 0, stream)
        st.sync()

    step(64)
    for i in range(81):
        step(1 + i)
        if i % 10 == 0:
            step(100)
    assert ctx.graph_stats() == (1, 0)          # recorded at the ninth
    step(100)
    assert ctx.graph_stats() == (1, 1)
    st.close()
    ctx.close()


def test_more_windows_than_graphs():
    """32 windows have graphs; another gets one only once 64 steps had no use for theirs.  The logits are those of direct launches."""
    runs = []
    for on in (False, True):
        cfg, ids, ctx = _context()
        ctx.set_graphs(on)
        stream = torch.cuda.Stream(device=DEV)
        st = wd.State(ctx, ids)
        logits = torch.zeros(128, cfg["V"], device=DEV)
        st.set_taps(logits=logits)
        torch.cuda.synchronize()
        got, stats = [], []
        for windows in (list(range(1, 41)), list(range(40, 0, -1)), [50] * 90):
            for i in range(0, len(windows), 10):
                _steps(st, windows[i:i + 10], stream)
                got.append(logits.clone())      # of the ten's last step, and what larger ones left behind
            stats.append(ctx.graph_stats())
        runs.append((got, stats))
        st.close()
        ctx.close()
    assert all(torch.equal(a, b) for a, b in zip(runs[0][0], runs[1][0], strict=True))
    assert runs[0][1] == [(0, 0)] * 3
    # 1 to 32 recorded, then replayed.  Window 32, the first of those to be used for the last time, was step 54 of 88 (each ten has
    # one of 64 active before it): step 119, the 28th of the window of 50, gets its place
    assert runs[1][1] == [(32, 0), (32, 32), (33, 32 + 90 - 28)]


def test_bf16_steps_synced_one_by_one():
    """A caller that waits for every step: the steps recorded with nothing queued, and those replayed, are the ones launched directly."""
    runs = []
    for on in (False, True):
        cfg, ids, ctx = _context(**BF16)
        ctx.set_graphs(on)
        stream = torch.cuda.Stream(device=DEV)
        st = wd.State(ctx, ids)
        outs = []
        for _ in range(40):
            st.step(8, 100, 20, 1, 1, stream)
            outs.append(st.sync())
        runs.append((st.read(0)["ids"], outs, ctx.graph_stats()))
        st.close()
        ctx.close()
    assert np.array_equal(runs[0][0], runs[1][0])
    for a, b in zip(runs[0][1], runs[1][1], strict=True):
        assert all(np.array_equal(a[n], b[n]) for n in ("n_unmasked", "positions", "token_ids", "confidence"))
    # two phases (of one and two key tiles) of a refresh and nineteen normal steps, the ninth of which is recorded
    assert runs[0][2] == (0, 0) and runs[1][2] == (2, 20)
