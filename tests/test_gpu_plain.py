"""CUDA-core kernels (fp32 models, index-list attention) at the edges of their tiles and of their dispatch, against float64."""
import numpy as np
import pytest
import torch

from paper_2601_20332_b200 import binding as wd
from paper_2601_20332_b200 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


# rows kernel: one piece, ragged pieces, k not a multiple of 4 (no vector loads), of 128, above 256, above one block of
# three 128-element loads; tile kernel, ragged in rows, columns and k; more rows than one grid holds
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("rows,n,k", [(1, 1, 5), (8, 16, 256), (9, 17, 64), (130, 101, 257), (33, 70, 388), (17, 36, 900),
                                      (1100, 1030, 36), (1031, 1024, 260), (524289, 3, 5)])
def test_gemm_plain_edges(dtype, rows, n, k):
    g = torch.Generator(device=DEV).manual_seed(rows * 7 + n)
    x = torch.randn(rows, k, device=DEV, generator=g).to(dtype)
    w = torch.randn(n, k, device=DEV, generator=g).to(dtype)
    y = wd.op_gemm(x, w, wd.WD_GEMM_PLAIN)
    ref = x.double() @ w.double().T
    # products of bf16 values are exact in fp32; k fp32 additions (and roundings of the products) of terms whose absolute
    # values sum to |x| |w|^T
    bound = (k + 1) * 2.0 ** -24 * (x.double().abs() @ w.double().abs().T)
    assert ((y.double() - ref).abs() <= bound + 1e-30).all()


# tiles filled through registers: k odd, rows that start off a 16-byte boundary, ragged rows,
# columns and k, a last row tile with one row, a first one with 33
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("rows,n,k,shift", [(1100, 1030, 35, 0), (257, 2100, 255, 0), (640, 1030, 256, 1),
                                            (33, 8200, 687, 0), (129, 4097, 18, 3)])
def test_gemm_plain_unaligned(dtype, rows, n, k, shift):
    g = torch.Generator(device=DEV).manual_seed(rows * 7 + n)
    x = torch.randn(rows * k + shift, device=DEV, generator=g).to(dtype)[shift:].view(rows, k)
    w = torch.randn(n * k + shift, device=DEV, generator=g).to(dtype)[shift:].view(n, k)
    y = wd.op_gemm(x, w, wd.WD_GEMM_PLAIN)
    bound = (k + 1) * 2.0 ** -24 * (x.double().abs() @ w.double().abs().T)         # as above
    assert ((y.double() - x.double() @ w.double().T).abs() <= bound + 1e-30).all()


# eight lanes per key with one to four 16-byte pieces per lane, fewer pieces than lanes, rows not a multiple of 16 bytes
# and rows above 512 bytes (a warp per key); key counts around the sixteen keys of a warp and the 128 of a block
@pytest.mark.parametrize("dtype,dh", [(torch.float32, 16), (torch.float32, 64), (torch.float32, 128), (torch.float32, 6),
                                      (torch.float32, 160), (torch.bfloat16, 64), (torch.bfloat16, 128), (torch.bfloat16, 20)])
@pytest.mark.parametrize("n_vis", [1, 15, 129, 300])
def test_attention_plain_edges(dtype, dh, n_vis):
    rows, Hq, Hkv, S = 3, 4, 2, 320
    g = torch.Generator(device=DEV).manual_seed(dh + n_vis)
    q = torch.randn(rows, Hq, dh, device=DEV, generator=g).to(dtype)
    k = torch.randn(Hkv, S, dh, device=DEV, generator=g).to(dtype)
    v = torch.randn(Hkv, dh, S, device=DEV, generator=g).to(dtype)
    vis = torch.randperm(S, device=DEV, generator=g)[:n_vis].to(torch.int32)
    out = wd.op_attention(q, k, v, vis).double()
    kk = k.double()[:, vis.long()].repeat_interleave(Hq // Hkv, 0)
    vv = v.double()[:, :, vis.long()].repeat_interleave(Hq // Hkv, 0)
    s = torch.einsum("rhd,hjd->rhj", q.double(), kk) / dh ** 0.5
    ref = torch.einsum("rhj,hdj->rhd", s.softmax(-1), vv)
    # scores up to about 5 in size with fp32 errors of dh * 2^-24 relative, __expf good to a few ulp of its argument's
    # size, sums of at most 300 terms: 1e-5 of the largest value; bf16 results are rounded to 8 bits on top
    tol = 1e-5 * float(v.abs().max()) + (2.0 ** -8 * ref.abs() if dtype == torch.bfloat16 else 0.0)
    assert ((out - ref).abs() <= tol).all()


# many blocks of few head dims (128 threads, a dim per warp): rows that are not 16-byte pieces, next to no keys, and both sides of
# the line between the two forms (2368 blocks, 8 keys for aligned rows)
@pytest.mark.parametrize("dtype,dh,rows,n_vis", [(torch.float32, 6, 592, 33), (torch.float32, 6, 591, 33), (torch.float32, 16, 700, 1),
                                                 (torch.float32, 32, 700, 8), (torch.float32, 32, 700, 9), (torch.bfloat16, 20, 600, 130),
                                                 (torch.bfloat16, 2, 1200, 5)])
def test_attention_plain_many_small_blocks(dtype, dh, rows, n_vis):
    Hq, Hkv, S = 4, 2, 136
    g = torch.Generator(device=DEV).manual_seed(dh + n_vis)
    q = torch.randn(rows, Hq, dh, device=DEV, generator=g).to(dtype)
    k = torch.randn(Hkv, S, dh, device=DEV, generator=g).to(dtype)
    v = torch.randn(Hkv, dh, S, device=DEV, generator=g).to(dtype)
    vis = torch.randperm(S, device=DEV, generator=g)[:n_vis].sort().values.to(torch.int32)
    out = wd.op_attention(q, k, v, vis).double()
    kk = k.double()[:, vis.long()].repeat_interleave(Hq // Hkv, 0)
    vv = v.double()[:, :, vis.long()].repeat_interleave(Hq // Hkv, 0)
    ref = torch.einsum("rhj,hdj->rhd", (torch.einsum("rhd,hjd->rhj", q.double(), kk) / dh ** 0.5).softmax(-1), vv)
    tol = 1e-5 * float(v.abs().max()) + (2.0 ** -8 * ref.abs() if dtype == torch.bfloat16 else 0.0)        # as above
    assert ((out - ref).abs() <= tol).all()


def test_fp32_steps_replayed_from_graphs():
    """Queued fp32 steps are recorded and replayed; the generation is the one that direct launches give."""
    cfg = synth.get_config("tiny", P=100, G=60)            # the visible range grows across a key tile (128) on the way
    w = synth.make_weights(cfg, DEV)
    ids = synth.make_prompts(cfg)
    S = ids.shape[1]
    runs = []
    for on in (False, True):
        ctx = wd.Context(cfg, w, 1, S, S, cfg["A"])
        ctx.set_graphs(on)
        st = wd.State(ctx, ids)
        _, steps, tokens = st.generate(cfg["A"], cfg["B"], cfg["R"], cfg["T"], cfg["k"], 0, torch.cuda.Stream(device=DEV))
        assert tokens == 60
        runs.append((st.read(0)["ids"], ctx.graph_stats()))
        st.close()
        ctx.close()
    assert np.array_equal(runs[0][0], runs[1][0])
    assert runs[0][1] == (0, 0) and runs[1][1][1] > 15


# fp32 steps with the element-wise kernels inside the projections (few rows) and beside them, against the float64 oracle: refresh
# and normal steps of one row to a few hundred, on either side of the four-row form's, the eight-row form's and the tiles' limits;
# grouped heads, rotation pairs that do not fill a group of columns' block, head_dim not a multiple of 4 (separate kernels),
# reduction lengths below one load, of one and of several blocks.  1e-5: rounding of fp32 sums over up to 900 terms, two blocks deep.
@pytest.mark.parametrize("over,batch,P,A,B", [
    (dict(), 1, 1, 1, 2), (dict(Hkv=2), 2, 33, 5, 7), (dict(), 1, 60, 24, 1), (dict(d=100, Hq=5, Hkv=1, dh=12, F=36, V=257), 3, 19, 4, 3),
    (dict(d=64, Hq=3, Hkv=3, dh=6, F=900, V=130), 1, 40, 9, 4), (dict(d=900, Hq=2, Hkv=1, dh=36, F=772, V=300), 1, 9, 3, 2),
    (dict(), 2, 120, 16, 40)])
def test_fused_rows_steps(over, batch, P, A, B):
    from wd_harness import Parity
    cfg = synth.get_config("tiny", **over)
    ids = synth.make_prompts(cfg, batch=batch, P=P, G=A + B + 6)
    p = Parity(cfg, synth.make_weights(cfg, DEV, gain_jitter=0.1), ids)
    for _ in range(4):
        r = p.step(A, B, 3, 2, 1, tol_layer=1e-5, tol_attn=1e-5)
        assert r["worst"]["logits"] <= 1e-5
    p.check_state_mirror()
    p.close()
