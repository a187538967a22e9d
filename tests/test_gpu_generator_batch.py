"""Training gradients of a large batch against the oracle.

The bias gradients leave 128 partial sums per image row of the batch: 4928 rows
need more than the 622,592 doubles that the buffer once held whatever the
batch. The rollout's history, allocated behind it, stays as it was. Bounds as
in the other gradient test (operands rounded to bfloat16 on both sides): loss
1e-4, every tensor 5e-3 in the 2-norm.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CIN = 6


@pytest.mark.parametrize("batch,ny,nz", [(64, 77, 128)])
def test_gradients_of_many_rows(batch, ny, nz):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import generator as og
    from paper_2103_08246_gb300 import binding, build, inputs
    build.build()
    w = inputs.generator_params(11, 128, 0, CIN, out_scale=1.0, bias_std=0.1)
    p = og.unflatten(w.astype(np.float32).astype(np.float64), 128, 0, CIN)
    rng = np.random.default_rng(5)
    qt, qp, tg = (rng.standard_normal((batch, ny, nz, 3)).astype(np.float32).astype(np.float64) for _ in range(3))
    gen = binding.Generator(ny, nz, blocks=0, in_channels=CIN, batch=batch)
    gen.set_params(w)
    gen.set_norm([0.0] * 3, [1.0] * 3, [1.0] * 3)
    gen.rollout_init(*rng.standard_normal((2, 3, ny, nz)))
    before = gen.history()
    loss = gen.grad(qt, qp, tg)
    g = gen.grads()
    after = gen.history()
    gen.close()
    assert all(np.array_equal(a, b) for a, b in zip(before, after))
    loss_ref, ref = og.loss_and_grads(p, [og.make_input(qt[b], qp[b], CIN) for b in range(batch)], list(tg), bf16=True)
    assert abs(loss - loss_ref) <= 1e-4 * loss_ref
    ref = og.flatten(ref)
    off = 0
    for n in (9 * 128 * CIN, 128, 9 * 3 * 128, 3):
        a, r = g[off:off + n], ref[off:off + n]
        assert np.linalg.norm(a - r) <= 5e-3 * np.linalg.norm(r), (off, n)
        off += n
    assert off == g.size
