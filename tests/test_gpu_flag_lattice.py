"""The structural update on lattices at the edges of its patches against the
oracle (automatic differentiation of the spring-network energy, FP64).

The lattice form splits the vertices into up to 16 patches with a halo of two
points; lattices whose largest patch no longer fits shared memory (beyond
84 x 84) take the list form. Sizes: no interior vertices, fewer rows than
patches would need, uneven splits, the sizes in use, the last lattice of the
patch form and the first of the list form.

Tolerance: 1e-9 of each quantity's largest value after three steps, the bound
of every FP64 parity test here. The double-single forces round at 2^-47 of
their terms (the stretching term k_s against forces of about 1e-2 k_s strain:
relative errors near 1e-11), integrated over at most 60 sub-steps.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("ns,nt,span", [(2, 2, 1.0), (2, 9, 1.0), (5, 3, 0.5), (9, 9, 1.0), (13, 7, 0.5), (17, 17, 1.0),
                                        (23, 41, 1.0), (33, 33, 1.0), (84, 84, 1.0), (85, 85, 1.0)])
def test_structure_matches_oracle(ns, nt, span):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle.solver import OracleSolver
    from paper_2103_08246_gb300 import binding, build, inputs
    build.build()
    wl = inputs.small(48, 16, 32, lx=3.0, ly=1.0, lz=2.0, re=200.0, flag_on=True, flag_x_le=0.5, flag_ns=ns, flag_nt=nt,
                      flag_len=1.0, flag_span=span, bending=0.02, dt=4e-3)
    noise = inputs.initial_noise(wl, amp=0.05)
    gpu, ora = binding.Solver(wl, binding.IBM_FP64, noise=noise), OracleSolver(wl, noise)
    gpu.step(3)
    ora.run(3)
    for name, g, o in zip("XVF", gpu.flag(), (ora.X, ora.V, ora.F_flag)):
        err = np.abs(g - o).max() / max(np.abs(o).max(), 1e-30)
        assert err <= 1e-9, (name, err)
    gpu.close()
