"""FP64 grids too small to fill the GPU (csrc/dgpe_engine.cuh, the fine variants): chunks of three to five points,
narrow blocks, radices up to five, and chunk scans cut to the chunks' reach; against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

SMALL = [(3, (32, 32, 32)), (3, (64, 40, 48)), (3, (96, 32, 80)), (2, (128, 160)), (2, (96, 160)), (2, (256, 192)),
         (2, (320, 384)), (2, (384, 512))]


def _solver(dim, n, h, nu, g, gdd, dt, imag, kernel=None, **kw):
    from paper_1601_04640_gb300 import build as gbuild
    from paper_1601_04640_gb300 import dgpe
    gbuild.build()
    return dgpe.Solver(dim, n, h, nu, g, gdd, dt, imag, True, kernel, **kw)


@pytest.mark.parametrize("imag", [True, False])
@pytest.mark.parametrize("kt", [1e-3, 0.0125, 0.3, 3.0, 30.0])
@pytest.mark.parametrize("case", range(len(SMALL)))
def test_solve_reach(case, kt, imag):
    """The solves alone (no trap, no interactions), from chunks that reach one neighbour to ones that reach the line's end."""
    from paper_1601_04640_gb300 import dgpe, synth
    dim, n = SMALL[case]
    h, nu = (0.2,) * dim, (0.0,) * dim
    dt = kt * 4 * 0.04
    psi0 = synth.gaussian_state(n, h, (1.0, 0.8, 1.2)[:dim], 0.3, 7)
    op = oracle.Params(dim=dim, n=n, h=h, nu=nu, g=0, gdd=0, dt=dt, imag=imag, kernel="none")
    with _solver(dim, n, h, nu, 0.0, 0.0, dt, imag, dgpe.DGPE_KERNEL_NONE) as s:
        s.set_psi(psi0)
        s.step(2)
        psi = s.get_psi()
    ref = oracle.step(op, psi0, 0, 2)
    e = np.linalg.norm(psi - ref) / np.linalg.norm(ref)
    # 2 dim solves: some 30 roundings of increments up to 4 kt times the state
    tol = 2 * dim * 30 * (1 + 4 * kt) * 2.0 ** -53
    print(n, kt, imag, "rel L2", e, "tol", tol)
    assert e < tol


@pytest.mark.parametrize("form", ["imag", "imag real state", "real"])
@pytest.mark.parametrize("case", range(len(SMALL)))
def test_step_and_observables(case, form):
    from paper_1601_04640_gb300 import synth
    dim, n = SMALL[case]
    imag, real_psi = form != "real", form == "imag real state"
    h, nu, g, gdd, dt = (0.2, 0.25, 0.3)[:dim], (1.0, 1.3, 0.8)[:dim], 40.0, 8.0, 1e-3
    psi0 = synth.gaussian_state(n, h, nu, 0.0 if real_psi else 0.01, 3)
    if real_psi:
        psi0 = psi0.real.astype(complex)
    op = oracle.Params(dim=dim, n=n, h=h, nu=nu, g=g, gdd=gdd, dt=dt, imag=imag,
                       kernel="dipolar3d" if dim == 3 else "quasi2d", qd=0.5)
    with _solver(dim, n, h, nu, g, gdd, dt, imag, real_psi=real_psi) as s:
        s.set_psi(psi0)
        s.step(9)  # one run of several steps and single ones
        psi, o = s.get_psi(), s.observables()
    ref = oracle.step(op, psi0, 0, 9)
    r = oracle.observables(op, ref, 9)
    e = np.linalg.norm(psi - ref) / np.linalg.norm(ref)
    print(n, form, "rel L2", e, "energy", o["energy"] / r["energy"] - 1)
    assert e < 9 * 100 * 2.0 ** -53
    for k in ("norm", "energy", "mu", "kin", "pot", "contact", "rms_r"):
        assert abs(o[k] - r[k]) <= 1e-11 * abs(r[k])
