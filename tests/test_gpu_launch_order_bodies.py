"""The forcing's kernels placed behind the one before them (programmatic stream
serialisation), beside the structural update on its own stream: several solvers
with bodies replayed at once, and the outflow plane where the x factor's
segments end.

Eulerian bars without a flag add in no order, so solvers side by side give the
bits of one alone. Markers add in the order of their atomics: FP64 sides differ
by rounding, which eleven steps leave below 1e-10 of the largest value (the
bound for one solver's run against another's); FP32 2e-5, as against the oracle.
The oracle comparisons use the bounds of the parity tests.
"""
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _precision(binding, name):
    return {"fp64": binding.IBM_FP64, "fp32": binding.IBM_FP32, "mixed": binding.IBM_MIXED}[name]


@pytest.mark.parametrize("precision", ["fp64", "fp32", "mixed"])
@pytest.mark.parametrize("bodies", ["eulerian", "markers", "flag"])
def test_solvers_with_bodies_side_by_side(precision, bodies):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2103_08246_gb300 import binding, build, inputs
    build.build()
    kw = dict(bars_on=True, bar_x=1.0)
    if bodies == "eulerian":
        kw["bar_forcing"] = "eulerian"
    if bodies == "flag":
        kw.update(flag_on=True, flag_x_le=2.0, flag_ns=17, flag_nt=17, flag_len=1.0, flag_span=1.0)
    h = 1 / 16
    wl = inputs.small(56, 32, 32, lx=56 * h, ly=32 * h, lz=32 * h, dt=2e-3, **kw)
    noise = inputs.initial_noise(wl, amp=0.1)

    def advance(s):
        for n in (1, 4, 6):
            s.step(n)
        return [np.array(a) for a in s.fields()] + ([np.array(a) for a in s.flag()[:2]] if wl.flag_on else [])
    prec = _precision(binding, precision)
    alone = binding.Solver(wl, prec, noise=noise)
    want = advance(alone)
    alone.close()
    solvers = [binding.Solver(wl, prec, noise=noise) for _ in range(4)]
    with ThreadPoolExecutor(len(solvers)) as pool:
        got = list(pool.map(advance, solvers))
    tol = 0.0 if bodies == "eulerian" else (1e-10 if precision == "fp64" else 2e-5)
    for s, fields in zip(solvers, got):
        for a, b in zip(fields, want):
            assert np.abs(a - b).max() <= tol * max(np.abs(b).max(), 1.0)
        s.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nx,afx", [(64, 64), (65, 64), (66, 64), (129, 64), (33, 32), (34, 32), (49, 24), (17, 16)])
def test_outflow_plane_at_segment_ends(precision, nx, afx):
    """u has nx - 1 unknowns along x, v and w nx: the last segment of each
    advances the outflow plane once, whether it is full, empty or of one plane."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle.solver import OracleSolver
    from paper_2103_08246_gb300 import binding, build, inputs
    build.build()
    wl = inputs.small(nx, 16, 16)
    noise = inputs.initial_noise(wl, amp=0.1)
    gpu = binding.Solver(wl, _precision(binding, precision), noise=noise, tiles={"afx_planes": afx})
    ora = OracleSolver(wl, noise)
    gpu.step(3)
    ora.run(3)
    for name, g, o in zip("uvw", gpu.fields(), ora.fields()):
        scale = np.abs(o).max() if precision == "fp64" else 1.0
        assert np.abs(g - o).max() <= (1e-9 if precision == "fp64" else 2e-5) * scale, name
    gpu.close()
