"""The constant-coefficient, chunked Crank-Nicolson solve of the FP32 bulk
(csrc/dgpe_lines.cuh): its algebra and its reach rules against the oracle's
Thomas solve in FP64 on the CPU, and the kernels on the GPU over line lengths
and kt = dt / (4 h^2) from one neighbouring chunk to the table form."""
import numpy as np
import pytest

import oracle


def _rule(kt, cl, tpl):
    """alpha, -2 kt m, the chunk reach dl (0: tables) and the in-chunk reach J."""
    m = 2.0 / (1.0 + 2.0 * kt + np.sqrt(1.0 + 4.0 * kt + 0j))
    al = kt * m
    rho = abs(al ** cl)
    dl = next((d for d in range(1, min(4, tpl) + 1) if rho ** d <= 2.0 ** -32 * (1.0 - rho)), 0)
    J = 1
    while J < cl and abs(al) ** (J + 1) > 2.0 ** -32:
        J += 1
    return al, -2.0 * kt * m, dl, J


def _solve(psi, kt, cl):
    n = psi.size
    tpl = n // cl
    al, m2, dl, J = _rule(kt, cl, tpl)
    assert dl > 0
    l = 2.0 * psi - np.concatenate(([0], psi[:-1])) - np.concatenate((psi[1:], [0]))
    y = l.reshape(tpl, cl).astype(complex)
    for i in range(1, cl):
        y[:, i] += al * y[:, i - 1]
    end, pc = y[:, -1].copy(), al ** cl
    for q in range(tpl):
        inflow = 0.0
        for j in range(max(0, q - dl), q):
            inflow = pc * inflow + end[j]
        y[q, :J] += al ** np.arange(1, J + 1) * inflow
    for i in range(cl - 2, -1, -1):
        y[:, i] += al * y[:, i + 1]
    end = y[:, 0].copy()
    for q in range(tpl):
        inflow = 0.0
        for j in range(min(tpl - 1, q + dl), q, -1):
            inflow = pc * inflow + end[j]
        y[q, cl - J:] += (al ** np.arange(1, J + 1))[::-1] * inflow
    u0 = y[0, 0]
    for q in range(min(dl, tpl)):
        y[q, :J] -= al ** np.arange(1, J + 1) * (al * pc ** q * u0)
    return psi + m2 * y.reshape(-1)


@pytest.mark.parametrize("imag", [True, False])
@pytest.mark.parametrize("tau", [0.002, 0.0125, 0.05, 0.25, 0.6, 1.2])
@pytest.mark.parametrize("n,cl", [(32, 16), (64, 16), (512, 16), (48, 12), (384, 12), (40, 10), (320, 10)])
def test_chunked_constant_form_matches_thomas(n, cl, tau, imag):
    kt = tau if imag else 1j * tau
    al, m2, dl, _ = _rule(kt, cl, n // cl)
    if dl == 0:
        pytest.skip("taken by the table form")
    rng = np.random.default_rng(n + int(1000 * tau))
    psi = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    p = oracle.Params(dim=2, n=(n, 32), h=(0.5, 0.5), nu=(0, 0), g=0, gdd=0, dt=tau, imag=imag, kernel="none")
    ref = oracle.cn_axis(p, np.ascontiguousarray(np.broadcast_to(psi, (32, n))), 0)[5]
    # four sums are cut at 2^-32 of a chunk's end value, at most 4 max|psi| / (1 - |alpha|)^2
    tol = 4 * abs(m2) * 4 / (1 - abs(al)) ** 2 * 2.0 ** -32 * np.max(np.abs(psi)) + 1e-14 * np.max(np.abs(psi))
    assert np.max(np.abs(_solve(psi, kt, cl) - ref)) <= tol


GPU_GRIDS = [(3, (32, 512, 40)), (3, (48, 40, 384)), (3, (64, 320, 32)), (2, (80, 32)), (2, (512, 192)), (2, (40, 512))]


@pytest.mark.gpu
@pytest.mark.parametrize("imag", [True, False])
@pytest.mark.parametrize("kt", [0.0125, 0.2, 0.8, 30.0])
@pytest.mark.parametrize("case", range(len(GPU_GRIDS)))
def test_gpu_cn_regimes(case, kt, imag):
    from paper_1601_04640_gb300 import build as gbuild
    from paper_1601_04640_gb300 import dgpe, synth
    gbuild.build()
    dim, n = GPU_GRIDS[case]
    h, nu = (0.2,) * dim, (0.0,) * dim
    dt = kt * 4 * 0.04
    psi0 = synth.gaussian_state(n, h, (1.0, 0.8, 1.2)[:dim], 0.3, 7)
    op = oracle.Params(dim=dim, n=n, h=h, nu=nu, g=0, gdd=0, dt=dt, imag=imag, kernel="none")
    with dgpe.Solver(dim, n, h, nu, 0.0, 0.0, dt, imag, False, dgpe.DGPE_KERNEL_NONE) as s:
        s.set_psi(psi0)
        s.step(2)
        psi = s.get_psi()
    ref = oracle.step(op, psi0, 0, 2)
    e = np.linalg.norm(psi - ref) / np.linalg.norm(ref)
    tol = max(1e-5, 4 * (1 + 4 * kt) * 2.0 ** -24)
    print(n, kt, imag, "rel L2", e, "tol", tol)
    assert e < tol
