"""q/k/v projections whose epilogue rotates the heads and writes the cache (many rows, whole tiles), against the oracle."""
import pytest

from paper_2601_20332_b200 import binding as wd
from paper_2601_20332_b200 import synth
from wd_harness import Parity

pytestmark = pytest.mark.gpu
DEV = "cuda"


# 911 rows in four token tiles of 240 x 39 weight tiles = 156 units for 74 CTA pairs.  26 heads, and 25, whose last tile holds
# one head; a second sequence whose rows start at an odd offset, so that its chunks of 16 tokens straddle the two sequences and
# start at positions that are no multiple of eight; one sequence alone of 897 rows, whose last chunk is one token.
@pytest.mark.parametrize("heads,batch,cut", [(26, 2, 41), (25, 2, 40), (26, 1, 0)])
def test_rope_epilogue(heads, batch, cut):
    cfg = synth.get_config("llada8b", L=1, d=256, Hq=heads, Hkv=heads, dh=128, F=512, V=1000, P=420 if batch == 2 else 841, G=100)
    w = synth.make_weights(cfg, DEV, gain_jitter=0.1)
    ids = synth.make_prompts(cfg, batch=batch)
    if cut:
        ids[1, cfg["P"] - cut:] = cfg["mask_id"]
    par = Parity(cfg, w, ids)
    launches = []
    for _ in range(2):                      # a refresh through the epilogue, a normal step that reads the cache it wrote
        assert par.step(16, 40, 4, 2, 1) is not None
        launches.append(par.log[-1]["info"]["n_launches"])
    assert par.log[0]["info"]["n_rows"] == (952 - cut if batch == 2 else 897)
    assert launches[0] == launches[1] - 1   # no rotation kernel


# grouped heads, in launches of whole units that do not fill two rounds: 38 query, two key and two value tiles of two heads x two token
# tiles = 84 units for 74 pairs; 57 heads over 3, where the last tile of every segment holds one head, and 600 rows of two sequences
@pytest.mark.parametrize("Hq,Hkv,batch,P", [(76, 4, 1, 244), (57, 3, 2, 244)])
def test_rope_epilogue_grouped_heads(Hq, Hkv, batch, P):
    cfg = synth.get_config("llada8b", L=1, d=1024, Hq=Hq, Hkv=Hkv, dh=128, F=512, V=1000, P=P, G=100)
    ids = synth.make_prompts(cfg, batch=batch)
    par = Parity(cfg, synth.make_weights(cfg, DEV, gain_jitter=0.1), ids)
    launches = []
    for _ in range(2):
        assert par.step(16, 40, 4, 2, 1) is not None
        launches.append(par.log[-1]["info"]["n_launches"])
    assert par.log[0]["info"]["n_rows"] == batch * (P + 56)
    assert launches[0] == launches[1] - 1   # no rotation kernel
    par.close()


# q/k/v of 16384 columns or more, enough units of 512 tokens for two rounds: the epilogue before a second accumulator.  24576 columns
# without grouping, and 18432 of 128 query heads over 8
@pytest.mark.parametrize("Hq,Hkv", [(64, 64), (128, 8)])
def test_rope_epilogue_wide(Hq, Hkv):
    cfg = synth.get_config("llada8b", L=1, d=256, Hq=Hq, Hkv=Hkv, dh=128, F=512, V=1000, P=544 if Hkv == 64 else 1046, G=100)
    par = Parity(cfg, synth.make_weights(cfg, DEV, gain_jitter=0.1), synth.make_prompts(cfg))
    launches = []
    for _ in range(2):
        assert par.step(16, 40, 4, 2, 1) is not None
        launches.append(par.log[-1]["info"]["n_launches"])
    assert par.log[0]["info"]["n_rows"] == cfg["P"] + 56
    assert launches[0] == launches[1] - 1   # no rotation kernel
    par.close()
