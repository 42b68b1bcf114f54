"""The CTA-group GEMM (sgd_kernel_gemm variant 0) against the oracle, at one shape at least per group,
tile width and epilogue that the rule picks there on 152 SMs (asserted), with ragged last tiles in
M, N and K.
Bounds: fp16 results the rounding of the result plus fp32 accumulation; fp32 results
accumulation alone, 2^-23 x sqrt(K) x the terms' norm with a factor of 8 for the tensor cores'
truncation."""
import math

import numpy as np
import pytest
import torch

from oracle import denoiser as odn
from test_gpu_kernels import _check_f16, _f, _rand

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2609_29505_gb300 import binding, build
    build.build()
    binding.lib()
    return binding


def _rows(rng, M):
    """Up to 200 rows to compare: the first and last, a tile's edge, others at random."""
    r = np.unique(np.r_[0, 127, 128, M - 1, rng.choice(M, min(M, 200), replace=False)])
    return r[r < M]


def _assert_tile(B, M, N, K, e, want):
    """The (group, columns) that the rule picks, where the GPU has the SMs it was written down for."""
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        assert B.sgd_kernel_gemm_tile(M, N, K, e) == want


# shape: tile of the plain epilogues and of the residual ones.  One CTA of width 64 (one row and 8
# columns; ragged; several waves), 128, 256; pairs of 160, 192, 224, 256 and, with a long K, 128
SHAPES = {(1, 8, 8): ((1, 64), (1, 64)), (128, 1000, 688): ((1, 64), (1, 64)), (257, 8200, 264): ((1, 64), (1, 64)),
          (333, 4096, 2056): ((1, 128), (1, 128)), (4012, 3024, 144): ((1, 256), (1, 128)),
          (1427, 1632, 464): ((2, 160), (1, 64)), (3073, 824, 592): ((2, 192), (1, 64)),
          (1034, 2936, 872): ((2, 224), (1, 64)), (2852, 2696, 800): ((2, 256), (2, 256)),
          (333, 4096, 8200): ((2, 128), (2, 128))}
# the residual epilogue's other widths, and two sizes of whole projections
RESIDUAL = {(3231, 3856, 264): (1, 256), (516, 3864, 584): (2, 160), (780, 3104, 792): (2, 192),
            (779, 3680, 1008): (2, 224), (2048, 1280, 5120): (2, 160), (4096, 4096, 4096): (2, 224)}
CASES = [(e, *s, t[e in ("delta", "gate")]) for s, t in SHAPES.items() for e in ("f16", "f32", "gelu", "delta", "gate")]
CASES += [(e, *s, t) for s, t in RESIDUAL.items() for e in ("delta", "gate")]


def test_every_width_is_among_the_cases():
    widths = {(1, 64), (1, 128), (1, 256), (2, 128), (2, 160), (2, 192), (2, 224), (2, 256)}
    for kinds in (("f16", "f32", "gelu"), ("delta", "gate")):
        assert {c[4] for c in CASES if c[0] in kinds} == widths


@pytest.mark.parametrize("epi,M,N,K,tile", CASES)
def test_group_plain_and_residual(B, epi, M, N, K, tile):
    rng = np.random.default_rng(M + N + K)
    A, W = _rand(rng, (M, K)).cuda(), _rand(rng, (N, K), 1 / math.sqrt(K)).cuda()
    rows = _rows(rng, M)
    want = odn.linear(_f(A[rows]), _f(W))
    tol = 8 * 2.0 ** -23 * math.sqrt(K) + 1e-6  # of results of unit scale
    if epi in ("delta", "gate"):
        h = torch.from_numpy(rng.standard_normal((M, N)).astype(np.float32)).cuda()
        h0, cache = _f(h[rows]), torch.zeros(M, N, dtype=torch.float16, device="cuda")
        e = B.sgd_epilogue_args(kind=B.EPI_DELTA, h=h.data_ptr(), ldh=N, cache=cache.data_ptr(), ld_cache=N)
        if epi == "gate":  # samples of 100 rows: one or two per 32-row warp
            g = torch.from_numpy(rng.standard_normal((-(-M // 100), N)).astype(np.float32)).cuda()
            e.gate, e.ld_gate, e.rows_per_batch = g.data_ptr(), N, 100
            want = want * _f(g)[rows // 100]
        _assert_tile(B, M, N, K, e, tile)
        B.sgd_kernel_gemm(A, W, M, N, K, e)
        np.testing.assert_allclose(_f(h[rows]), h0 + want, rtol=2e-6, atol=6 * tol)
        _check_f16(cache[rows], want, extra_abs=6 * tol)
    else:
        out = torch.full((M, N), 7.0, dtype=torch.float32 if epi == "f32" else torch.float16, device="cuda")
        kind = {"f16": B.EPI_F16, "f32": B.EPI_F32, "gelu": B.EPI_GELU}[epi]
        e = B.sgd_epilogue_args(kind=kind, out=out.data_ptr(), ldo=N)
        _assert_tile(B, M, N, K, e, tile)
        B.sgd_kernel_gemm(A, W, M, N, K, e)
        if epi == "f32":
            np.testing.assert_allclose(_f(out[rows]), want, rtol=2e-6, atol=6 * tol)
        else:
            # the activations' fast exponential: 2^-21 relative
            _check_f16(out[rows], odn.gelu_tanh(want) if epi == "gelu" else want, extra_abs=6 * tol + 2e-6)
    torch.cuda.synchronize()
    assert B.sgd_kernel_status() == 0


@pytest.mark.parametrize("M,N,K,tile", [(64, 688, 256, (1, 128)), (383, 32, 8, (1, 128)), (3217, 2624, 8, (1, 256)),
                                        (272, 3592, 856, (2, 224)), (1040, 3456, 784, (2, 256))])
@pytest.mark.parametrize("act", [0, 1])
def test_group_gated(B, M, N, K, tile, act):
    rng = np.random.default_rng(M + N + K + act)
    A, W = _rand(rng, (M, K)).cuda(), _rand(rng, (2 * N, K), 1 / math.sqrt(K)).cuda()
    out = torch.full((M, N), 7.0, dtype=torch.float16, device="cuda")
    e = B.sgd_epilogue_args(kind=B.EPI_GATED, out=out.data_ptr(), ldo=N, act=act)
    _assert_tile(B, M, N, K, e, tile)
    B.sgd_kernel_gemm(A, W, M, N, K, e)
    rows = _rows(rng, M)
    u = odn.linear(_f(A[rows]), _f(W))
    want = u[:, :N] * odn.gelu_erf(u[:, N:]) if act else odn.silu(u[:, :N]) * u[:, N:]
    _check_f16(out[rows], want, extra_abs=2e-5 * float(np.abs(want).max()))
    assert B.sgd_kernel_status() == 0


@pytest.mark.parametrize("dh", [64, 128])
@pytest.mark.parametrize("M,heads,K,tile", [(1, 1, 16, (1, 128)), (100, 7, 72, (1, 128)), (4146, 23, 16, (1, 256)),
                                            (3382, 11, 776, (2, 256))])
def test_group_rope(B, M, heads, K, tile, dh):
    rng = np.random.default_rng(M + heads + K + dh)
    N, tokens, half = 3 * heads * dh, 50, dh // 2
    A, W = _rand(rng, (M, K)).cuda(), _rand(rng, (N, K), 1 / math.sqrt(K)).cuda()
    ang = rng.standard_normal((tokens, half)).astype(np.float32)
    cos, sin = (torch.from_numpy(f(ang)).cuda() for f in (np.cos, np.sin))
    out = torch.full((M, N), 7.0, dtype=torch.float16, device="cuda")
    e = B.sgd_epilogue_args(kind=B.EPI_ROPE, out=out.data_ptr(), ldo=N, rope_cos=cos.data_ptr(),
                            rope_sin=sin.data_ptr(), rope_tokens=tokens, d_head=dh, rope_cols=2 * heads * dh)
    _assert_tile(B, M, N, K, e, tile)
    B.sgd_kernel_gemm(A, W, M, N, K, e)
    u = odn.linear(_f(A), _f(W)).reshape(M, 3 * heads, dh)
    c, s = _f(cos)[np.arange(M) % tokens][:, None], _f(sin)[np.arange(M) % tokens][:, None]
    r = u[:, :2 * heads]
    rot = np.concatenate([r[..., :half] * c - r[..., half:] * s, r[..., half:] * c + r[..., :half] * s], -1)
    want = np.concatenate([rot, u[:, 2 * heads:]], 1).reshape(M, N)
    _check_f16(out, want, extra_abs=2e-5)
    assert B.sgd_kernel_status() == 0
