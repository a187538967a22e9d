"""The flag's interpolation in a uniform stream is free of bias.

With u = U everywhere and the flag at rest the first step's fluid force is
U dv / dt times the sum of the 27 weights, which is 1. Each weight rounds by
half a unit in the last place at most, either way: over some 1500 vertices at
incommensurate places the mean stays below a quarter of a unit (its noise is
about a hundredth). Weights that all carry the rounding of one constant, 1/6,
shift it by three quarters.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision", ["fp64", "fp32", "mixed"])
def test_weights_sum_to_one(precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import flag
    from paper_2103_08246_gb300 import binding, build, inputs
    build.build()
    wl = inputs.small(48, 32, 32, lx=3.0, ly=2.0, lz=2.0, flag_on=True, flag_x_le=1.03, flag_ns=41, flag_nt=37, flag_len=1.01,
                      flag_span=1.07, dt=2e-3)
    prec = {"fp64": binding.IBM_FP64, "fp32": binding.IBM_FP32, "mixed": binding.IBM_MIXED}[precision]
    gpu = binding.Solver(wl, prec)
    gpu.step(1)
    F = np.array(gpu.flag()[2])
    gpu.close()
    dv = flag.FlagMesh(41, 37, wl.flag_len, wl.flag_span, 1.0, 1.0, 1.0).area * (wl.lx / wl.nx)
    total = F[:, 0] * wl.dt / dv
    assert np.abs(F[:, 1:]).max() == 0.0
    unit = np.finfo(np.float64 if precision == "fp64" else np.float32).eps
    assert np.abs(total - 1.0).max() <= 8 * unit
    assert abs(np.mean(total - 1.0)) <= 0.25 * unit, np.mean(total - 1.0) / unit
