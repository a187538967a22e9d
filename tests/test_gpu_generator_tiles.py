"""The generator's forward pass at the edges of its tiling, against the oracle.

One to three tiles of 128 or 256 pixels per CTA, counts just below and above
the number of SMs, a row of three tiles, the smallest plane. Operands are
rounded to bfloat16 on both sides, so the bounds are those of the other
forward test: 2e-3 of the largest output (one operand whose rounding flips),
1e-4 of it in the mean.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

BLOCKS, CIN = 2, 6


@pytest.mark.parametrize("ny,nz,batch", [(3, 128, 1), (19, 128, 8), (20, 128, 8), (40, 128, 8), (52, 384, 1),
                                         (3, 256, 1), (76, 256, 1), (77, 256, 1), (160, 256, 1), (57, 256, 4), (114, 512, 1)])
def test_forward_matches_oracle(ny, nz, batch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import generator as og
    from paper_2103_08246_gb300 import binding, build, inputs
    build.build()
    w = inputs.generator_params(11, 128, BLOCKS, CIN, block_scale=0.5, out_scale=1.0, bias_std=0.1)
    p = og.unflatten(w.astype(np.float32).astype(np.float64), 128, BLOCKS, CIN)
    rng = np.random.default_rng(ny)
    qt, qp = (rng.standard_normal((batch, ny, nz, 3)).astype(np.float32).astype(np.float64) for _ in range(2))
    gen = binding.Generator(ny, nz, blocks=BLOCKS, in_channels=CIN, batch=batch)
    gen.set_params(w)
    d = gen.forward(qt, qp)
    gen.close()
    for b in {0, batch - 1}:
        ref, _ = og.forward(p, og.make_input(qt[b], qp[b], CIN), bf16=True)
        err = np.abs(d[b] - ref)
        scale = np.abs(ref).max()
        assert err.max() <= 2e-3 * scale, (b, err.max(), scale)
        assert err.mean() <= 1e-4 * scale, (b, err.mean(), scale)
