"""dgpe_pass_flops counts the form of the Crank-Nicolson solve that runs (csrc/dgpe_lines.cuh: difference, two
recurrences, three fix-ups of J sites of a chunk, last product)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("imag", [True, False])
@pytest.mark.parametrize("kt", [0.0125, 0.8, 30.0])
def test_constant_form_and_tables(kt, imag):
    from paper_1601_04640_gb300 import build as gbuild
    from paper_1601_04640_gb300 import dgpe
    gbuild.build()
    n, h, cl = (64, 128, 64), (0.2, 0.2, 0.2), 16
    with dgpe.Solver(3, n, h, (1.0, 1.0, 1.0), 10.0, 5.0, kt * 4 * 0.04, imag, False) as s:
        names = [dgpe.load().dgpe_pass_name(s.h, i).decode() for i in range(dgpe.dgpe_launches_per_step(s.h))]
        flops = dict(zip(names, (dgpe.load().dgpe_pass_flops(s.h, i) for i in range(len(names)))))
    k = kt if imag else 1j * kt
    al = abs(k * 2.0 / (1.0 + 2.0 * k + np.sqrt(1.0 + 4.0 * k + 0j)))
    dl = next((d for d in range(1, 5) if al ** (cl * d) <= 2.0 ** -32 * (1.0 - al ** cl)), 0)
    J = 1
    while J < cl and al ** (J + 1) > 2.0 ** -32:
        J += 1
    m, tpl = (4, n[1] // cl) if imag else (8, n[1] // cl)
    per = 6 + 3 * m + (3 * J + 2 * dl) * m / cl if dl else (28 + 10 * np.log2(tpl) / cl if imag else 52 + 28 * np.log2(tpl) / cl)
    sites = n[0] * n[1] * n[2]
    print(kt, imag, "dl", dl, "J", J, "per site", flops["cn_y"] / sites, per)
    assert abs(flops["cn_y"] / sites - per) < 1e-9 * per
    assert all(f > 0 for f in flops.values())
