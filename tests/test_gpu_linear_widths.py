"""sc_linear_forward where the tile width and the list of row tiles are chosen on
the device: 64-column tiles with more K steps than stages, sequences without
rows before, between and after others, the most sequences whose tiles are
counted out and one more, and widths that leave 64- and 192-column tiles."""
import math

import numpy as np
import pytest
import torch

from oracle import encoder as enc
from test_gpu_encoder import _bf16, _t_bf16, sc  # noqa: F401

pytestmark = pytest.mark.gpu

CASES = [
    # B, L, rows, N, K
    (1, 200, [200], 768, 3072),
    (1, 200, None, 640, 64),
    (5, 256, [0, 0, 256, 0, 129], 2304, 128),
    (3, 129, [0, 0, 0], 256, 64),
    (128, 140, [(37 * b) % 141 for b in range(128)], 384, 128),
    (129, 140, [(53 * b) % 141 for b in range(129)], 384, 128),
]


@pytest.mark.parametrize("B,L,rows,N,K", CASES)
def test_linear_widths(sc, B, L, rows, N, K):  # noqa: F811
    rng = np.random.default_rng(B + L + N + K)
    A = _bf16(rng.standard_normal((B * L, K)))
    W = _bf16(rng.standard_normal((N, K)) / math.sqrt(K))
    bias = rng.standard_normal(N).astype(np.float32)
    out = torch.full((B * L, N), float("nan"), dtype=torch.float32, device="cuda")
    n = np.array(rows if rows is not None else [L] * B, np.int32)
    sc.linear_forward(_t_bf16(A), _t_bf16(W), B=B, L=L,
                      rows=torch.from_numpy(n).cuda() if rows is not None else None,
                      bias=torch.from_numpy(bias).cuda(), out=out, out_f32=True)
    got = out.cpu().numpy().astype(np.float64).reshape(B, L, N)
    want = enc.linear(A, W, bias).reshape(B, L, N)
    used = np.arange(L)[None, :] < n[:, None]
    # fp32 sums of K exact products: the bar of the other fp32 outputs
    np.testing.assert_allclose(got[used], want[used], rtol=0, atol=1e-4 * np.abs(want).max())
    assert np.isnan(got[~used]).all(), "rows past the sequence were written"


@pytest.mark.parametrize("gelu,out_f32", [(False, True), (True, False), (True, True)])
def test_linear_residual_of_four_chunks(sc, gelu, out_f32):  # noqa: F811
    """Gathered rows keep 256-column tiles: a write-back warp takes four chunks of
    the residual, two loaded before the product is there and two on the way."""
    rng = np.random.default_rng(3)
    B, L, N, K, n = 2, 150, 384, 128, np.array([150, 131], np.int32)
    A = _bf16(rng.standard_normal((B * L, K)))
    W = _bf16(rng.standard_normal((N, K)) / math.sqrt(K))
    R = _bf16(rng.standard_normal((B * L, N)))
    gidx = np.stack([rng.permutation(L) for _ in range(B)]).astype(np.int32)
    out = torch.full((B * L, N), float("nan"), device="cuda",
                     dtype=torch.float32 if out_f32 else torch.bfloat16)
    sc.linear_forward(_t_bf16(A), _t_bf16(W), B=B, L=L, rows=torch.from_numpy(n).cuda(),
                      gidx=torch.from_numpy(gidx).cuda(), gelu=gelu, res=_t_bf16(R),
                      res_gathered=True, out=out, out_f32=out_f32)
    got = out.float().cpu().numpy().astype(np.float64)
    for b in range(B):
        src = b * L + gidx[b, :n[b]]
        y = enc.linear(A[src], W, np.zeros(N))
        y = (enc.gelu(y) if gelu else y) + R[src]
        # bf16 out: half an ulp, 2^-9 |y|, and as much again for the fp32 part
        tol = (1e-4 * np.abs(y).max(), 0) if out_f32 else (1e-4, 2.0 ** -8)
        np.testing.assert_allclose(got[b * L:b * L + n[b]], y, atol=tol[0], rtol=tol[1])
        assert np.isnan(got[b * L + n[b]:(b + 1) * L]).all()
