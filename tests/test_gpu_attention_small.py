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
