"""The factor that the FP64 transforms leave to the x solve, against the oracle:
a factor of 4 for each direction of at most 256 points, none for a longer one,
so planes with either, both or neither direction beyond 256, and the smallest
planes. FP64 bound 1e-9 relative, as in the other parity tests.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nx,ny,nz", [(6, 4, 4), (6, 8, 256), (6, 512, 16), (6, 16, 512), (4, 512, 512)])
def test_pressure_matches_oracle(nx, ny, nz):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle.solver import OracleSolver
    from paper_2103_08246_gb300 import binding, build, inputs
    build.build()
    wl = inputs.small(nx, ny, nz, dt=-1.0, cfl=0.3)
    noise = inputs.initial_noise(wl, amp=0.1)
    gpu, ora = binding.Solver(wl, binding.IBM_FP64, noise=noise), OracleSolver(wl, noise)
    gpu.step(2)
    ora.run(2)
    for name, g, o in zip("uvwp", gpu.fields(), ora.fields()):
        if name == "p":
            g, o = g - g.mean(), o - o.mean()
        assert np.abs(g - o).max() <= 1e-9 * np.abs(o).max(), name
    gpu.close()
