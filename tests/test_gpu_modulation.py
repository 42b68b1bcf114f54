"""AdaLN modulation of every active branch in one launch, where its weights are many enough for
the kernel that streams them through shared memory (two DiT-XL/2-wide blocks: 4 segments of
3456 x 1152), at batch sizes 2 to 9: 2 and 8 rows stream, 1 and 9 do not.  One step against the
oracle, relative L2 as for every step (fp16 operands)."""
import numpy as np
import pytest
import torch

from oracle import denoiser as odn
from paper_2609_29505_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 2, 8, 9])
def test_wide_modulation(batch):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2609_29505_gb300 import binding, build
    build.build()
    cfg = synth.get_config("dit").with_(name="dit_wide", n_blocks=2, batch=batch, n_tokens=16, T=1, horizons=[1])
    w = synth.make_weights(cfg, "cuda")
    inp = synth.make_inputs(cfg, "cpu")
    m = binding.Denoiser(cfg, w)
    m.set_schedule(1, [1] * cfg.n_units, synth.block_groups(cfg))
    out = torch.empty(batch, cfg.n_out_tokens, cfg.out_channels, device="cuda")
    m.step(inp.z0.cuda(), out, 700.0, 1, class_ids=inp.class_ids.cuda())
    m.check_device()
    m.close()
    want = odn.denoise_full(cfg, odn.to_numpy_weights(w), inp.z0.numpy(), 700.0, class_ids=inp.class_ids.numpy())
    got = out.cpu().numpy()
    assert np.linalg.norm(got - want) <= 5e-3 * np.linalg.norm(want)
