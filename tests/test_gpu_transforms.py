"""The pressure solve's transforms at every radix split and at the edges of
their rules against the oracle: lines of 4 to 512 points in both directions
(one-pass planes in FP32, single directions in FP64, the radix-2 form beyond
256 points), square and uneven planes, an odd plane count; the mixed solve by
FFTs and on the tensor cores.

Two steps from noise excite every transverse mode. Bounds as in the other
parity tests: FP64 1e-9 relative; FP32 and mixed 2e-5 of the natural scales,
p 2e-4.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SHAPES = [(4, 4), (4, 256), (256, 4), (8, 16), (16, 8), (16, 16), (32, 64), (64, 32), (64, 64), (128, 32), (32, 128),
          (128, 128), (256, 128), (128, 256), (512, 4), (8, 512)]


def _check(ny, nz, precision, **kw):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle.solver import OracleSolver
    from paper_2103_08246_gb300 import binding, build, inputs
    build.build()
    wl = inputs.small(5, ny, nz)
    noise = inputs.initial_noise(wl, amp=0.1)
    gpu, ora = binding.Solver(wl, precision, noise=noise, **kw), OracleSolver(wl, noise)
    gpu.step(2)
    ora.run(2)
    fp64 = precision == binding.IBM_FP64
    for name, g, o in zip("uvwp", gpu.fields(), ora.fields()):
        if name == "p":
            g, o = g - g.mean(), o - o.mean()
        tol = 1e-9 * np.abs(o).max() if fp64 else (2e-4 if name == "p" else 2e-5)
        assert np.abs(g - o).max() <= tol, name
    gpu.close()


@pytest.mark.parametrize("precision", [0, 1, 2], ids=["fp64", "fp32", "mixed"])
@pytest.mark.parametrize("ny,nz", SHAPES)
def test_transforms_match_oracle(ny, nz, precision):
    _check(ny, nz, precision)


@pytest.mark.parametrize("n", [32, 64, 128, 256])
def test_tensor_core_solve_matches_oracle(n):
    _check(n, n, 2, tc_predictor=True)
