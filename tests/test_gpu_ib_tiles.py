"""Bar-marker forcing at the edges of the tile shapes against the oracle.

The tiles shrink with the transverse plane (16 x 16 down to 4 x 8 cells), the
plane's short sides cut them further, and FP64 spreads straight to the field
while FP32 sums in shared memory. One parity run per shape with bars and a
flag whose vertices lie across the periodic sides; bounds as in the other
parity tests (FP64 1e-9 relative; FP32 2e-5 of the natural scales).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("ny,nz", [(4, 8), (8, 4), (8, 32), (64, 16), (32, 32), (64, 64), (128, 64)])
def test_bars_match_oracle(precision, ny, nz):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle.solver import OracleSolver
    from paper_2103_08246_gb300 import binding, build, inputs
    build.build()
    h = 1.0 / 8.0
    wl = inputs.small(24, ny, nz, lx=24 * h, ly=ny * h, lz=nz * h, bars_on=True, bar_x=0.75, bar_mesh=0.5, bar_width=0.2,
                      flag_on=True, flag_x_le=1.25, flag_ns=7, flag_nt=9, flag_len=1.0, flag_span=1.0)
    noise = inputs.initial_noise(wl, amp=0.05)
    prec = binding.IBM_FP64 if precision == "fp64" else binding.IBM_FP32
    gpu, ora = binding.Solver(wl, prec, noise=noise), OracleSolver(wl, noise)
    gpu.step(3)
    ora.run(3)
    for name, g, o in zip("uvwp", gpu.fields(), ora.fields()):
        if name == "p":
            g, o = g - g.mean(), o - o.mean()
        scale = np.abs(o).max() if precision == "fp64" else 1.0
        tol = 1e-9 if precision == "fp64" else (2e-4 if name == "p" else 2e-5)
        assert np.abs(g - o).max() <= tol * scale, name
    gpu.close()
