"""The structural update on long, narrow lattices against the oracle.

The lattice form holds positions in fixed point, 2^49 per scaled unit (the
longest spring is 1/2 to 1 unit). Lattices of 257 points and more along a side
lie more than 128 units from their corner; up to 2176 x 2 points fit the
patches' shared memory. Sizes: the first past 128 units, square cells and
oblong ones (the scale follows the longest spring), along the chord and along
the span, up to 1000 points.

Tolerance: 1e-9 of each quantity's largest value after three steps, the bound
of every FP64 parity test here. The state's own rounding at the far end,
k_s 2^-53 x over the vertex mass for one sub-step (random over some twenty of
them), stays near 1e-10 of the vertex speeds at 1000 spacings.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("ns,nt,ds,dt", [(257, 3, 1 / 16, 1 / 16), (258, 17, 1 / 16, 1 / 16), (400, 9, 1 / 16, 1 / 16),
                                         (700, 9, 1 / 16, 1 / 16), (1000, 2, 1 / 16, 1 / 20), (321, 5, 1 / 32, 1 / 8),
                                         (17, 258, 1 / 32, 1 / 32)])
def test_long_lattice_matches_oracle(ns, nt, ds, dt):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle.solver import OracleSolver
    from paper_2103_08246_gb300 import binding, build, inputs
    build.build()
    length, span, h = (ns - 1) * ds, (nt - 1) * dt, 1 / 16
    nx = int(np.ceil(length / h)) + 16
    nz = 256 if span > 2.0 else 32
    wl = inputs.small(nx, 16, nz, lx=nx * h, ly=1.0, lz=nz * h, re=200.0, flag_on=True, flag_x_le=0.5, flag_ns=ns,
                      flag_nt=nt, flag_len=length, flag_span=span, bending=0.02, dt=4e-3)
    noise = inputs.initial_noise(wl, amp=0.05)
    gpu, ora = binding.Solver(wl, binding.IBM_FP64, noise=noise), OracleSolver(wl, noise)
    gpu.step(3)
    ora.run(3)
    for name, g, o in zip("XVF", gpu.flag(), (ora.X, ora.V, ora.F_flag)):
        err = np.abs(g - o).max() / max(np.abs(o).max(), 1e-30)
        assert err <= 1e-9, (name, err)
    gpu.close()
