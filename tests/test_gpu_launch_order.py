"""Kernels placed behind the one before them (programmatic stream
serialisation) wait for its results: steps of a grid whose kernels take a few
microseconds each, replayed as graphs by several solvers on their own streams
at once, give the same bits as one solver alone. No marker takes part (the
forcing adds in no fixed order), so every sum has a fixed order and the bound is zero.
"""
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision", ["fp64", "fp32", "mixed"])
@pytest.mark.parametrize("nx,ny,nz", [(9, 16, 32), (33, 32, 64), (48, 64, 128), (20, 256, 256)])
def test_solvers_side_by_side_match_one_alone(precision, nx, ny, nz):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2103_08246_gb300 import binding, build, inputs
    build.build()
    wl = inputs.small(nx, ny, nz, dt=-1.0, cfl=0.3)
    noise = inputs.initial_noise(wl, amp=0.1)
    prec = {"fp64": binding.IBM_FP64, "fp32": binding.IBM_FP32, "mixed": binding.IBM_MIXED}[precision]
    alone = binding.Solver(wl, prec, noise=noise)
    for n in (1, 4, 7):
        alone.step(n)
    want = [np.array(a) for a in alone.fields()]
    alone.close()
    solvers = [binding.Solver(wl, prec, noise=noise) for _ in range(4)]

    def advance(s):
        for n in (1, 4, 7):
            s.step(n)

    with ThreadPoolExecutor(len(solvers)) as pool:
        list(pool.map(advance, solvers))
    for s in solvers:
        for name, a, b in zip("uvwp", s.fields(), want):
            assert np.array_equal(a, b), name
        s.close()
