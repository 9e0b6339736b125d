"""Output and down projections whose epilogue adds to the residual stream (many rows, whole tiles), against the oracle."""
import pytest

from paper_2601_20332_b200 import synth
from wd_harness import TOL_ATTN, TOL_LAYER, Parity

pytestmark = pytest.mark.gpu
DEV = "cuda"


# 20 weight tiles of 256, the last one half empty (width 39 x 128), and seven token tiles = 140 units for 74 CTA pairs; 1593 rows in
# tiles of 240, the last of 153 rows, its last chunk of nine; two sequences; without taps of the blocks the second of two blocks
# takes the gathered active rows instead
@pytest.mark.parametrize("batch,block_taps", [(1, True), (2, True), (1, False)])
def test_resid_epilogue(batch, block_taps):
    P = 1537 if batch == 1 else 747
    cfg = synth.get_config("llada8b", L=2, d=39 * 128, Hq=2, Hkv=2, dh=128, F=256, V=500, P=P, G=100)
    w = synth.make_weights(cfg, DEV, gain_jitter=0.1)
    ids = synth.make_prompts(cfg, batch=batch)
    if batch == 2:
        ids[1, P - 13:] = cfg["mask_id"]
    par = Parity(cfg, w, ids, block_taps=block_taps, follow_rounded=block_taps)
    launches = []
    for _ in range(2):                      # a refresh through the epilogue, a normal step that reads the cache it wrote
        # block l: the tolerance of one block times sqrt(l + 1), and at most a tenth more than what the bfloat16 storage points
        # alone cost (random weights this wide: 1.1e-2 after the second block), as in the full-depth tests
        log = par.step(16, 40, 4, 2, 1, envelope=lambda l: (TOL_LAYER * (l + 1) ** 0.5, TOL_ATTN * (l + 1) ** 0.5))
        launches.append(log["info"])
        if block_taps:
            assert all(a <= 1.10 * b for a, b in zip(log["curve"]["layer"], log["curve"]["layer_format"]))
    assert launches[0]["n_rows"] == 1593 and launches[0]["n_rows"] % 16 == 9
    if block_taps:                          # no kernel that adds the down projection for the taps
        assert launches[0]["n_launches"] == launches[1]["n_launches"] - 2
    par.close()
