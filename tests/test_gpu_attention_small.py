"""Attention shapes that impl 0 gives to the kernel with one query tile per CTA (key tiles of 64):
edges of its tiles in queries and keys, every head dimension, rows that need a rescale, and
queries and keys that end inside a warp.  Against the oracle's attention; relative L2 as in
test_gpu_kernels (fp16 operands, P in fp16)."""
import numpy as np
import pytest
import torch

from oracle import denoiser as odn
from test_gpu_kernels import _f, _rand

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dh", [64, 72, 128])
@pytest.mark.parametrize("bsz,H,nq,nkv", [(1, 1, 1, 1), (2, 3, 33, 63), (1, 2, 128, 64), (2, 2, 129, 65),
                                          (8, 16, 258, 258), (2, 4, 160, 77), (10, 16, 97, 200)])
@pytest.mark.parametrize("growing", [False, True])
def test_small_attention(bsz, H, nq, nkv, dh, growing):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2609_29505_gb300 import binding as B, build
    build.build()
    rng = np.random.default_rng(bsz * 1000 + nq + nkv + dh)
    hs = 80 if dh == 72 else dh
    q, k, v = (torch.zeros(bsz, n, H, hs, dtype=torch.float16) for n in (nq, nkv, nkv))
    for t in (q, k, v):
        t[..., :dh] = _rand(rng, t.shape[:3] + (dh,))
    if growing:  # row maxima grow along the keys: O is rescaled
        k[..., :dh] *= torch.linspace(0.2, 6.0, nkv)[None, :, None, None]
    o = torch.full((bsz, nq, H, dh), 7.0, dtype=torch.float16, device="cuda")
    dev = [t.cuda() for t in (q, k, v)]
    B.sgd_kernel_attention_hs(dev[0], H * hs, dev[1], dev[2], H * hs, hs, o, H * dh, bsz, nq, nkv, H, dh)
    torch.cuda.synchronize()
    flat = [_f(t[..., :dh].reshape(t.shape[0], t.shape[1], H * dh)) for t in (q, k, v)]
    want = odn.attention(*flat, H).reshape(bsz, nq, H, dh)
    err = np.linalg.norm(_f(o) - want) / np.linalg.norm(want)
    assert err < 1.5e-3, err
    assert B.sgd_kernel_status() == 0


# Shapes of the dispatch rule's own table that go to the kernel of one query tile.
@pytest.mark.parametrize("bsz,H,nq,nkv,dh", [(2, 20, 1024, 77, 64), (16, 16, 258, 258, 64), (2, 16, 136, 136, 72),
                                             (10, 16, 97, 200, 128)])
def test_first_reference_covers_128_keys(bsz, H, nq, nkv, dh):
    """Probabilities are rounded to fp16 against the same reference as in the kernel of two query tiles
    (impl 3), a row's maximum over its first 128 keys, so that the results agree but for the
    order of the fp32 row sum: that moves a result by about 2^-22 before its rounding, across a
    rounding boundary (2^-10 apart, relative) for one in 2^11 of them, by 2^-10.5 on average then:
    2^-10.5 x sqrt(2^-11) = 1.6e-5 relative L2, allowed twice.  (A reference over 64 keys: 1.4e-4.)"""
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2609_29505_gb300 import binding as B, build
    build.build()
    rng = np.random.default_rng(nq + nkv + dh)
    hs = 80 if dh == 72 else dh
    q, k, v = (torch.zeros(bsz, n, H, hs, dtype=torch.float16, device="cuda") for n in (nq, nkv, nkv))
    for t in (q, k, v):
        t[..., :dh] = _rand(rng, t.shape[:3] + (dh,)).cuda()
    got = []
    for impl in (0, 3):
        o = torch.full((bsz, nq, H, dh), 7.0, dtype=torch.float16, device="cuda")
        B.sgd_kernel_attention_hs(q, H * hs, k, v, H * hs, hs, o, H * dh, bsz, nq, nkv, H, dh, impl=impl)
        got.append(_f(o).astype(np.float64))
    assert np.linalg.norm(got[0] - got[1]) <= 3.2e-5 * np.linalg.norm(got[1])
    assert B.sgd_kernel_status() == 0
