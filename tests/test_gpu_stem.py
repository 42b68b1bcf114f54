"""The patch stems through one step of a one-block U-ViT-shaped model against the oracle, relative L2
as for every step (fp16 operands)."""
import numpy as np
import pytest
import torch

from oracle import denoiser as odn
from paper_2609_29505_gb300 import synth

pytestmark = pytest.mark.gpu


def _step(cfg, samples):
    """One step on the GPU; its output and the oracle's for the given samples of the batch."""
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2609_29505_gb300 import binding, build
    build.build()
    w = synth.make_weights(cfg, "cuda")
    inp = synth.make_inputs(cfg, "cpu")
    m = binding.Denoiser(cfg, w)
    m.set_schedule(1, [1] * cfg.n_units, synth.block_groups(cfg))
    out = torch.empty(cfg.batch, cfg.n_out_tokens, cfg.out_channels, device="cuda")
    m.step(inp.z0.cuda(), out, 700.0, 1, class_ids=inp.class_ids.cuda())
    m.check_device()
    m.close()
    want = odn.denoise_full(cfg.with_(batch=len(samples)), odn.to_numpy_weights(w), inp.z0[samples].numpy(), 700.0,
                            class_ids=inp.class_ids[samples].numpy())
    return out[samples].cpu().numpy(), want


def test_more_token_rows_than_a_grid_dimension_holds():
    """528384 token rows: more than 65535 blocks of 8."""
    cfg = synth.get_config("uvit_small").with_(name="uvit_rows", n_blocks=1, n_skips=0, d=64, n_heads=1, d_ff=128,
                                               batch=2048, n_tokens=258, T=1, horizons=[1])
    got, want = _step(cfg, [0, 1, 1024, 2047])
    assert np.linalg.norm(got - want) <= 5e-3 * np.linalg.norm(want)


@pytest.mark.parametrize("d_in", [8, 16, 24, 12])
def test_patch_widths(d_in):
    """Weight rows in registers (8, 16 channels), read as vectors (24) and one by one (12); 201 token rows
    end inside a block's 8, and 576 channels inside the second block's 512."""
    cfg = synth.get_config("uvit_small").with_(name="uvit_patch%d" % d_in, n_blocks=1, n_skips=0, d=576, n_heads=9,
                                               d_ff=128, n_tokens=67, d_in=d_in, T=1, horizons=[1])
    got, want = _step(cfg, [0, 1, 2])
    assert np.linalg.norm(got - want) <= 5e-3 * np.linalg.norm(want)
