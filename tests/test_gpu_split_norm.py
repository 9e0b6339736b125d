"""Steps of few rows, whose RMSNorm leaves 1 / rms to the consumers of the projections (four blocks to a row)."""
import pytest

from paper_2601_20332_b200 import synth
from wd_harness import Parity

pytestmark = pytest.mark.gpu


# one row; a width that does not fill the blocks' last warp; head_dim 64, 128 and 12 (single rotation pairs, ragged V tiles), grouped
# heads; 128 rows, the last that takes it, and 129 at a refresh; widths below and above its range (2048 and 4096 inside)
@pytest.mark.parametrize("over,P,A,B", [
    (dict(d=2112, Hq=4, Hkv=2, dh=128), 1, 1, 1), (dict(d=2048, Hq=16, Hkv=16, dh=64), 96, 20, 12),
    (dict(d=3584, Hq=16, Hkv=4, dh=12), 97, 24, 8), (dict(d=4096, Hq=2, Hkv=1, dh=128), 20, 33, 40),
    (dict(d=1984, Hq=4, Hkv=4, dh=64), 20, 9, 4), (dict(d=4160, Hq=4, Hkv=4, dh=64), 20, 9, 4)])
def test_split_norm_steps(over, P, A, B):
    cfg = synth.get_config("tiny", dtype="bf16", F=320, V=512, **over)
    ids = synth.make_prompts(cfg, batch=1, P=P, G=A + B + 6)
    p = Parity(cfg, synth.make_weights(cfg, "cuda", gain_jitter=0.1), ids)
    # heads of 12 dims, input rows of 3584: scores of size sqrt(3584) * 0.02^2 * 3584 / sqrt(12) ~ 25 before the softmax, which the
    # rounding of q and k (2^-9 each, 12 terms of random sign) moves by 25 * 2^-9 * sqrt(2 / 12) ~ 2e-2, and the weights by as much
    # (1.9e-2 with a block to a row, too)
    tol_attn = 3e-2 if cfg["dh"] == 12 else 2e-2
    for _ in range(4):
        p.step(A, B, 3, 2, 1, tol_attn=tol_attn)
    p.check_state_mirror()
    p.close()
