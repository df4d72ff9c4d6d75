"""The warp-per-tile x-row passes of the FP32 bulk (csrc/dgpe_rows*.cu) and the
strided transforms of every line length against the oracle: every supported
row length, row counts that fill no whole tile, both modes, a real state, and
exponents from the short series to the library functions."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

# second sizes whose pairs of rows are no multiple of a tile's
GRIDS = [(32, 40), (64, 48), (128, 40), (256, 32), (512, 32), (48, 96), (96, 40), (192, 384), (384, 192), (40, 32),
         (80, 160), (160, 320), (320, 80)]


@pytest.mark.parametrize("form", ["imag", "imag real state", "real"])
@pytest.mark.parametrize("n", GRIDS)
def test_rows_of_every_length(n, form):
    from paper_1601_04640_gb300 import build as gbuild
    from paper_1601_04640_gb300 import dgpe, synth
    gbuild.build()
    imag, real_psi = form != "real", form == "imag real state"
    h, nu, g, gdd = (0.2, 0.25), (1.0, 1.3), 40.0, 8.0
    psi0 = synth.gaussian_state(n, h, nu, 0.0 if real_psi else 0.01, 3)
    if real_psi:
        psi0 = psi0.real.astype(complex)
    vmax = 0.5 * ((n[0] * 0.1) ** 2 + (1.3 * n[1] * 0.125) ** 2)
    # largest exponent of a step: within 1/8, within 1 (2), beyond
    for top in (0.1, 0.9, 6.0):
        dt = top / vmax
        op = oracle.Params(dim=2, n=n, h=h, nu=nu, g=g, gdd=gdd, dt=dt, imag=imag, kernel="quasi2d", qd=0.5)
        with dgpe.Solver(2, n, h, nu, g, gdd, dt, imag, False, real_psi=real_psi) as s:
            s.set_psi(psi0)
            s.step(3)
            psi = s.get_psi()
        ref = oracle.step(op, psi0, 0, 3)
        e = np.linalg.norm(psi - ref) / np.linalg.norm(ref)
        # three steps of some 40 roundings (2^-24) each, and of the exponent (2^-24 of it)
        tol = 3 * (40 + 4 * top) * 2.0 ** -24
        print(n, form, top, "rel L2", e, "tol", tol)
        assert e < tol


@pytest.mark.parametrize("nx", [64, 96, 320])
def test_rows_modes_of_the_reverse_step(nx):
    """Phi_d alone, the real input field and the conjugated solve (the state at an address the bulk copies
    can start at, and eight bytes behind one)."""
    import ctypes
    import torch
    from paper_1601_04640_gb300 import build as gbuild
    from paper_1601_04640_gb300 import dgpe, synth
    gbuild.build()
    n, h, nu, dt = (nx, 40, 32), (0.2, 0.25, 0.3), (1.0, 1.2, 0.8), 2e-3
    psi0 = synth.gaussian_state(n, h, nu, 0.01, 5)
    G0 = synth.gaussian_state(n, h, (0.8, 1.0, 1.1), 0.05, 6)
    op = oracle.Params(dim=3, n=n, h=h, nu=nu, g=40.0, gdd=8.0, dt=dt, imag=False, kernel="dipolar3d")
    Gr = oracle.step_adjoint(op, psi0, G0, 0)[0]
    with dgpe.Solver(3, n, h, nu, 40.0, 8.0, dt, False, False) as s:
        for off in (0, 1):
            a = torch.empty(psi0.size + 2, dtype=torch.complex64, device="cuda")
            b = torch.empty_like(a)
            p, g = a[off:off + psi0.size], b[off:off + psi0.size]
            p.copy_(torch.from_numpy(psi0.astype(np.complex64)).reshape(-1))
            g.copy_(torch.from_numpy(G0.astype(np.complex64)).reshape(-1))
            dgpe.dgpe_step_adjoint(s.h, p.data_ptr(), g.data_ptr(), 0, 0)
            got = g.cpu().numpy().reshape(Gr.shape)
            e = np.linalg.norm(got - Gr) / np.linalg.norm(Gr)
            print(nx, off, "rel L2", e)
            assert e < 120 * 2.0 ** -24
