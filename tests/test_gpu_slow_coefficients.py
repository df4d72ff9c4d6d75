"""FP32 bulk at time steps whose Crank-Nicolson coefficients decay too slowly for the constant form (kt = dt / (4 h^2)
above some 8 in imaginary and 4 in real time): with dipoles, the x pass is then the block-wide one fed by bulk copies
(k_p1_pipe, power-of-two nx) or the one-block-per-tile one (other lengths, a real state), and the solves along y and z
read their coefficients from tables (csrc/dgpe_cols.cu)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

# nx from 32 to 512 and two lengths that are no power of two; second sizes that fill no whole tile of rows
GRIDS = [(32, 40), (64, 40), (128, 48), (256, 96), (512, 40), (96, 40), (160, 512), (64, 32, 40), (512, 32, 32), (128, 40, 64)]


@pytest.mark.parametrize("form", ["imag", "imag real state", "real"])
@pytest.mark.parametrize("n", GRIDS)
def test_step_with_dipoles_at_large_kt(n, form):
    from paper_1601_04640_gb300 import build as gbuild
    from paper_1601_04640_gb300 import dgpe, synth
    gbuild.build()
    imag, real_psi, dim, kt = form != "real", form == "imag real state", len(n), 10.0
    h = (0.2, 0.22, 0.25)[:dim]
    dt = kt * 4 * h[-1] ** 2  # kt >= 10 along every axis
    # exponents of a step up to 0.1 (short series), 0.9 and 3 (library functions) at the corners
    for top in (0.1, 0.9, 3.0):
        w = (2 * top / dt / sum((0.5 * k * d) ** 2 for k, d in zip(n, h))) ** 0.5
        nu, g, gdd = (w,) * dim, 0.3 * top / dt, 0.1 * top / dt
        psi0 = synth.gaussian_state(n, h, (1.0, 0.8, 1.2)[:dim], 0.0 if real_psi else 0.01, 9)
        if real_psi:
            psi0 = psi0.real.astype(complex)
        op = oracle.Params(dim=dim, n=n, h=h, nu=nu, g=g, gdd=gdd, dt=dt, imag=imag,
                           kernel="dipolar3d" if dim == 3 else "quasi2d", qd=0.5)
        ref = oracle.step(op, psi0, 0, 3)
        for flags in (0, dgpe.DGPE_FLAG_P1_ONESHOT):
            with dgpe.Solver(dim, n, h, nu, g, gdd, dt, imag, False, real_psi=real_psi, flags=flags) as s:
                s.set_psi(psi0)
                s.step(3)
                psi = s.get_psi()
            e = np.linalg.norm(psi - ref) / np.linalg.norm(ref)
            # a step: some 40 roundings (2^-24), those of the exponent, and two units of the increments, up to 4 kt
            # times the state (kt of the finest axis)
            tol = 3 * (40 + 4 * top + 2 * (1 + 4 * dt / (4 * h[0] ** 2))) * 2.0 ** -24
            print(n, form, top, flags, "rel L2", e, "tol", tol)
            assert e < tol
