"""The attention kernel with two query tiles per CTA (where that takes fewer rounds over the SMs), against the oracle."""
import numpy as np
import pytest
import torch

from oracle import wd_oracle as wo
from paper_2601_20332_b200 import binding as wd
from paper_2601_20332_b200 import synth
from wd_harness import Parity

pytestmark = pytest.mark.gpu
DEV = "cuda"


# more than 148 (row tile, query head) items: an odd number of tiles (a CTA with one), a last tile of one row, one key tile,
# one key in the last tile, one below and one above a tile; grouped-query heads whose items pair across row tiles (7 per
# tile); packed heads (two and four per tile) with empty slots; scores whose row maxima grow by tens of units from tile to
# tile, so that the accumulated output is rescaled, and mild ones, where it is not; then both sides of the rule at an equal
# number of rounds (one tile per KV head: 64 and 65 rows over one key tile, 96 and 97 over two, three key tiles)
@pytest.mark.parametrize("rows,nv,Hq,Hkv,S,qs", [(257, 128, 64, 64, 136, 1.5), (300, 127, 64, 64, 128, 8.0),
                                                 (260, 129, 56, 8, 136, 8.0), (130, 1025, 84, 12, 1032, 8.0),
                                                 (640, 400, 32, 32, 400, 1.5), (33, 300, 320, 64, 304, 8.0),
                                                 (20, 700, 693, 99, 704, 1.5), (128, 1, 160, 160, 8, 1.5),
                                                 (64, 128, 160, 160, 128, 1.5), (65, 128, 160, 160, 128, 8.0), (96, 256, 160, 160, 256, 8.0),
                                                 (97, 256, 160, 160, 256, 1.5), (128, 257, 160, 160, 264, 8.0)])
def test_two_tiles_per_cta_vs_oracle(rows, nv, Hq, Hkv, S, qs):
    g = torch.Generator(device=DEV).manual_seed(rows + nv)
    q = (torch.randn(rows, Hq, 128, device=DEV, generator=g) * qs).to(torch.bfloat16)
    kc = torch.randn(Hkv, S, 128, device=DEV, generator=g).to(torch.bfloat16)
    kc *= torch.linspace(0.5, 2.0, S, device=DEV).to(torch.bfloat16)[None, :, None]        # later keys score higher
    vc = torch.randn(Hkv, S, 128, device=DEV, generator=g).to(torch.bfloat16)
    K = kc.double().cpu().numpy().transpose(1, 0, 2)[:nv]
    V = vc.double().cpu().numpy().transpose(1, 0, 2)[:nv]
    kc[:, nv:] = float("nan")                       # what must not be read as a value
    vc[:, nv:] = float("nan")
    out = wd.op_attention_tc(q, kc, vc.transpose(1, 2).contiguous(), nv).float().cpu().numpy().astype(np.float64)
    assert wd.op_status() == 0 and np.isfinite(out).all()
    ref, _ = wo.attention_rows(q.double().cpu().numpy(), K, V, Hq // Hkv)
    # P and the result rounded to bf16: as in test_attention_tc_kernel_vs_oracle
    assert np.abs(out - ref).max() / np.abs(ref).max() < 2e-2


# six, three and one query tiles of 16 heads: 160 single tiles, 96 pairs, CTAs beyond a shorter sequence's last pair leave at once
# and odd sequences end in half a pair; with grouped heads (five to a KV head) pairs cross row tiles
@pytest.mark.parametrize("Hq,Hkv", [(16, 16), (20, 4)])
def test_sequences_of_different_lengths(Hq, Hkv):
    cfg = synth.get_config("llada8b", L=1, d=256, Hq=Hq, Hkv=Hkv, dh=128, F=512, V=1000, P=650, G=80)
    w = synth.make_weights(cfg, DEV, gain_jitter=0.1)
    ids = synth.make_prompts(cfg, batch=3)
    ids[1, 300:] = cfg["mask_id"]
    ids[2, 50:] = cfg["mask_id"]
    par = Parity(cfg, w, ids)
    for _ in range(2):
        info = par.step(16, 40, 4, 2, 1)["info"]
    assert par.log[0]["info"]["n_rows"] == 706 + 356 + 106
    par.close()
