"""The error of the structural update's forces against 64 bits.

One step of one velocity-Verlet sub-step from rest: V = h (a0 + a1) / 2, so the
speeds give the forces back. The reference repeats the sub-step from the
solver's own X and fluid force, with FP64 forces by automatic differentiation
(error near 1e-16 k_s l) and every update rounded once, as the solver's fused
operations are.

Bound: the forces are unevaluated FP32 pairs, which hold 2^-49 of a length; ten
operations of half that, halved from squared to plain lengths and summed over
a vertex's eight springs, make about 2.2e-15 k_s l rms. 4e-15 leaves a factor
of two and stays below the 5e-15 of FP64 forces with one Newton step on an FP32
estimate of the square root.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("ns,nt,ds", [(9, 9, 1 / 8), (5, 23, 1 / 16), (17, 9, 1 / 16), (33, 17, 1 / 16), (9, 9, 0.11)])
def test_force_error(ns, nt, ds):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import flag
    from paper_2103_08246_gb300 import binding, build, inputs
    build.build()
    h, dt = 1 / 16, 1.8 / 126.5 * ds * 0.5
    nx = int(np.ceil((ns - 1) * ds / h)) + 16
    wl = inputs.small(nx, 32, 32, lx=nx * h, ly=2.0, lz=2.0, re=200.0, flag_on=True, flag_x_le=0.25, flag_ns=ns, flag_nt=nt,
                      flag_len=(ns - 1) * ds, flag_span=(nt - 1) * ds, pitch0=0.3, bending=0.005, dt=dt)
    mesh = flag.FlagMesh(ns, nt, wl.flag_len, wl.flag_span, wl.mass_ratio, wl.stretch, wl.bending)
    assert mesh.substeps(dt) == 1
    gpu = binding.Solver(wl, binding.IBM_FP64, noise=inputs.initial_noise(wl, amp=0.05))
    X = np.array(gpu.flag()[0])
    gpu.step(1)
    Xg, Vg, F = (np.array(a) for a in gpu.flag())
    gpu.close()
    L = np.longdouble
    l0, m = mesh.rest_lengths(X), mesh.mass[:, None]
    half = L(0.5 * dt)

    def acc(x):
        return np.where(mesh.free[:, None], (flag.elastic_forces(x, mesh, l0) + F) / m, 0.0)
    V = (half * L(acc(X))).astype(np.float64)
    X1 = (L(X) + L(dt) * L(V)).astype(np.float64)
    V = (L(V) + half * L(acc(X1))).astype(np.float64)
    assert np.abs(Xg - X1).max() <= 4e-16 * np.abs(X1).max()
    err = ((Vg - V) * m / dt / (wl.stretch * ds))[mesh.free]
    rms = float(np.sqrt(np.mean(err ** 2)))
    assert rms <= 4e-15, rms
