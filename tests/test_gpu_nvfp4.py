"""NVFP4 quantiser and GEMM at the edges of their work split (the common shapes are in test_gpu_ops.py)."""
import numpy as np
import pytest
import torch

from oracle import wd_oracle as wo
from paper_2601_20332_b200 import binding as wd

pytestmark = pytest.mark.gpu
DEV = "cuda"


def parts(raw, rows, k):
    up = lambda v: (v + 255) // 256 * 256
    codes = raw[: rows * k // 2].reshape(rows, k // 2)
    sf = raw[up(rows * k // 2): up(rows * k // 2) + rows * k // 16].reshape(rows, k // 16)
    g = raw[up(rows * k // 2) + up(rows * k // 16):][: 4 * rows].view(np.float32)
    grid = np.array([0.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 6.0])
    q = np.empty((rows, k))
    q[:, 0::2], q[:, 1::2] = [np.where(c & 8, -1.0, 1.0) * grid[c & 7] for c in (codes & 15, codes >> 4)]
    return q, torch.from_numpy(sf.copy()).view(torch.float8_e4m3fn).double().numpy(), g


# one block; a block count that is no multiple of a warp; more blocks than threads; an input that is not 16-byte aligned
@pytest.mark.parametrize("rows,k,shift", [(1, 16, 0), (3, 528, 0), (2, 16400, 0), (2, 784, 1)])
def test_quantise_edges_are_the_oracles_bytes(rows, k, shift):
    g = torch.Generator(device=DEV).manual_seed(k)
    x = torch.randn(rows * k + shift, device=DEV, generator=g).to(torch.bfloat16)[shift:].view(rows, k)
    q, sf, gr = parts(wd.op_nvfp4_quantize(x).cpu().numpy(), rows, k)
    rq, rs, rg = wo.nvfp4_quant_rows(x.float().cpu().numpy().astype(np.float64))
    np.testing.assert_array_equal(q, rq)
    np.testing.assert_array_equal(sf, rs)
    np.testing.assert_array_equal(gr, rg)


# a unit shared by many SMs, units that start and end inside a share, a grid cut down to the most slices (three units, one unit),
# whole units per SM because there are many, and two each on half of the SMs; two units in three equal shares, every share a fixed part of a unit, more sharers
# than units
@pytest.mark.parametrize("rows,n,k", [(34, 1000, 4096), (129, 2000, 1024), (5, 300, 16384), (600, 16000, 256), (5, 128, 16384),
                                      (34, 12288, 4096), (16, 4096, 1024), (64, 600, 8192), (16, 19200, 512)])
def test_gemm_edges(rows, n, k):
    g = torch.Generator(device=DEV).manual_seed(rows + n)
    x = torch.randn(rows, k, device=DEV, generator=g).to(torch.bfloat16)
    w = (torch.randn(n, k, device=DEV, generator=g) * 0.05).to(torch.bfloat16)
    xq, wq = wd.op_nvfp4_quantize(x), wd.op_nvfp4_quantize(w)
    y = wd.op_gemm_nvfp4(xq, wq, rows, n, k)
    assert torch.equal(y, wd.op_gemm_nvfp4(xq, wq, rows, n, k)) and wd.op_status() == 0
    ops = []
    for raw, m in ((xq, rows), (wq, n)):
        q, sf, gr = parts(raw.cpu().numpy(), m, k)
        ops.append(torch.from_numpy(q * np.repeat(sf, 16, 1) * gr[:, None].astype(np.float64)).to(DEV))
    ref = ops[0] @ ops[1].T
    # equal operands on both sides: fp32 accumulation only, as in test_gemm_nvfp4_vs_oracle
    assert float((y.double() - ref).abs().max()) <= 2e-5 * float(ref.abs().max())
