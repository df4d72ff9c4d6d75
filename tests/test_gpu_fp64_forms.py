"""Which FP64 form runs where (csrc/dgpe_engine.cuh: choose_cn_form, fine_sites), and that each gives the oracle's
step."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _dgpe():
    from paper_1601_04640_gb300 import build as gbuild
    from paper_1601_04640_gb300 import dgpe
    gbuild.build()
    return dgpe


def _names(dgpe, s):
    return [dgpe.load().dgpe_pass_name(s.h, i).decode() for i in range(dgpe.dgpe_launches_per_step(s.h))]


@pytest.mark.parametrize("n,serial", [((96, 96, 96), True), ((64, 80, 64), False)])
def test_real_time_without_dipoles_solves_lines_serially(n, serial):
    """From 8192 lines per axis the line-serial solve is the faster one in real time without dipoles, also on grids
    that take the small-grid passes (160^3: 711 against 1016 us a step); in imaginary time it is not (742 against
    647).  The form follows the mode."""
    dgpe = _dgpe()
    from paper_1601_04640_gb300 import synth
    h, nu, g, dt = (0.2, 0.25, 0.3), (1.0, 1.3, 0.8), 40.0, 1e-3
    psi0 = synth.gaussian_state(n, h, nu, 0.01, 3)
    ref, step = psi0, 0
    with dgpe.Solver(3, n, h, nu, g, 0.0, dt, False, True, dgpe.DGPE_KERNEL_NONE) as s:
        s.set_psi(psi0)
        for imag in (False, True, False):
            s.set_mode(imag)
            assert ("cn_x" in _names(dgpe, s)) == (serial and not imag)
            op = oracle.Params(dim=3, n=n, h=h, nu=nu, g=g, gdd=0.0, dt=dt, imag=imag, kernel="none")
            s.step(5)
            ref = oracle.step(op, ref, step, 5)
            step += 5
        e = np.linalg.norm(s.get_psi() - ref) / np.linalg.norm(ref)
        print(n, "rel L2", e)
        assert e < 15 * 100 * 2.0 ** -53


@pytest.mark.parametrize("form", ["imag", "imag real state", "real"])
@pytest.mark.parametrize("n", [(64, 64, 64), (128, 32, 64), (32, 128, 128), (128, 64, 64), (64, 128, 128)])
def test_power_of_two_boxes_on_both_sides_of_the_small_grid_passes(n, form):
    """2^18 and 2^19 sites take the small-grid passes, 2^20 the others; exponents on both sides of 1/8."""
    dgpe = _dgpe()
    from paper_1601_04640_gb300 import synth
    imag, real_psi = form != "real", form == "imag real state"
    h, nu, g, gdd, dt = (0.2, 0.25, 0.22), (1.0, 1.3, 0.8), 40.0, 8.0, 2e-3
    psi0 = synth.gaussian_state(n, h, nu, 0.0 if real_psi else 0.01, 3)
    if real_psi:
        psi0 = psi0.real.astype(complex)
    op = oracle.Params(dim=3, n=n, h=h, nu=nu, g=g, gdd=gdd, dt=dt, imag=imag, kernel="dipolar3d")
    with dgpe.Solver(3, n, h, nu, g, gdd, dt, imag, True, real_psi=real_psi) as s:
        s.set_psi(psi0)
        s.step(5)  # one run of several steps and a single one
        psi, o = s.get_psi(), s.observables()
    ref = oracle.step(op, psi0, 0, 5)
    r = oracle.observables(op, ref, 5)
    e = np.linalg.norm(psi - ref) / np.linalg.norm(ref)
    print(n, form, "rel L2", e, "energy", o["energy"] / r["energy"] - 1)
    assert e < 5 * 100 * 2.0 ** -53
    for k in ("norm", "energy", "mu", "kin", "pot", "contact", "rms_r"):
        assert abs(o[k] - r[k]) <= 1e-11 * abs(r[k])
