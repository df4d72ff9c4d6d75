"""FP64 Crank-Nicolson solves at large kt = dt / (4 h^2) on a smooth state, against the same solves in extended
precision (csrc/dgpe_fine.cu): the second difference must not cost more than the solve's own roundings.  A rounded
psi_{a-1} + psi_{a+1} leaves some 0.4 2^-53 psi at every site, which -2 kt A^-1 amplifies by 2 kt sqrt((1 + 2 kt) /
(1 + 4 kt)^1.5): 7 units of 2^-53 over the two solves at kt = 30 and 18 at kt = 100, beyond the bound below."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _solve(f, kt):
    """One substep of a line, long double complex."""
    T = np.clongdouble
    f, kt, n = f.astype(T), T(kt), f.size
    z = np.zeros(1, T)
    r = -2 * kt * (2 * f - np.concatenate((z, f[:-1])) - np.concatenate((f[1:], z)))
    m, y = [], []
    for a in range(n):
        m.append(1 / (1 + 2 * kt - (kt * kt * m[-1] if a else 0)))
        y.append((r[a] + (kt * y[-1] if a else 0)) * m[-1])
    for a in range(n - 2, -1, -1):
        y[a] = y[a] + kt * m[a] * y[a + 1]
    return f + np.array(y, T)


@pytest.mark.parametrize("imag", [True, False])
@pytest.mark.parametrize("kt", [30.0, 100.0])
@pytest.mark.parametrize("n", [(512, 512), (384, 512), (320, 512)])
def test_solves_on_a_smooth_state(n, kt, imag):
    from paper_1601_04640_gb300 import build as gbuild
    from paper_1601_04640_gb300 import dgpe
    gbuild.build()
    h = [14.0 / k for k in n]
    dt = kt * 4 * min(h) ** 2
    # a product state: the exact result is the product of the lines' results
    line = [np.exp(-0.3 * ((np.arange(k) - k // 2) * d) ** 2) for k, d in zip(n, h)]
    psi = (line[1][:, None] * line[0][None, :]).astype(complex)
    with dgpe.Solver(2, n, h, (0.0, 0.0), 0.0, 0.0, dt, imag, True, dgpe.DGPE_KERNEL_NONE) as s:
        s.set_psi(psi)
        s.step(1)
        got = s.get_psi()
    kts = [dt / (4 * d * d) for d in h]
    ex = [_solve(f, k if imag else 1j * k) for f, k in zip(line, kts)]
    ref = ex[1][:, None] * ex[0][None, :]
    if imag:
        ref = ref / np.sqrt(np.longdouble(h[0] * h[1]) * np.sum(ref.real ** 2 + ref.imag ** 2))
    e = float(np.sqrt(np.sum(np.abs(got - ref) ** 2) / np.sum(np.abs(ref) ** 2)) / 2.0 ** -53)
    # units of 2^-53: the product state and the scale (2), and per solve its last addition and the recurrences (0.8)
    # and alpha, which is off by 3 units at most (three roundings) and changes kt by sqrt(1 + 4 kt) of that, of which
    # a state with <k^2 h^2> = 0.3 h^2 feels 2 kt times that
    tol = 2 + sum(0.8 + 3 * np.sqrt(abs(1 + 4 * (k if imag else 1j * k))) * 2 * k * 0.3 * d * d for k, d in zip(kts, h))
    print(n, kt, imag, "units of 2^-53:", e, "tol", tol)
    assert e < tol
