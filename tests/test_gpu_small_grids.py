"""Launch shapes of the streamed kernels on small, short and uneven grids
against the oracle: planes per block of the explicit stage, the divergence and
the projection follow the grid (fewer planes on small grids, counts that do not
divide nx on larger ones), so x lengths around the chunk sizes, one plane more
or less than a chunk, and the smallest transverse planes of the run kernels.
CFL steps, so that the speed maxima of every block are used. Bounds as in the
other parity tests (FP64 1e-9 relative; FP32 2e-5 of the natural scales, p 2e-4).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nx,ny,nz", [(4, 8, 8), (5, 16, 32), (7, 32, 16), (16, 64, 32), (17, 16, 64), (33, 32, 128),
                                      (29, 8, 256), (67, 128, 32)])
def test_steps_match_oracle(precision, nx, ny, nz):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle.solver import OracleSolver
    from paper_2103_08246_gb300 import binding, build, inputs
    build.build()
    wl = inputs.small(nx, ny, nz, dt=-1.0, cfl=0.3)
    noise = inputs.initial_noise(wl, amp=0.1)
    prec = binding.IBM_FP64 if precision == "fp64" else binding.IBM_FP32
    gpu, ora = binding.Solver(wl, prec, noise=noise), OracleSolver(wl, noise)
    gpu.step(1)
    gpu.step(3)
    ora.run(4)
    assert abs(gpu.stats()["dt"] / ora.last_dt - 1.0) < (1e-12 if precision == "fp64" else 1e-5)
    for name, g, o in zip("uvwp", gpu.fields(), ora.fields()):
        if name == "p":
            g, o = g - g.mean(), o - o.mean()
        scale = np.abs(o).max() if precision == "fp64" else 1.0
        tol = 1e-9 if precision == "fp64" else (2e-4 if name == "p" else 2e-5)
        assert np.abs(g - o).max() <= tol * scale, name
    gpu.close()
