"""Host replay of the index arithmetic of the transforms whose stages are not those of test_fft_stage_indexing.py:
the solver's column tiles with a 12- or 20-point first stage (ct_radix_cols in csrc/dgpe_device.cuh), the warp-per-tile
rows (csrc/dgpe_rows.cuh) and the FP64 small grids (csrc/dgpe_fine.cu).  Every stage reads and writes every element of
every line exactly once, inside the tile, and every twiddle is the one the transform needs."""
import pytest

from test_fft_stage_indexing import ct_radix

LENGTHS = [32, 64, 128, 256, 512, 48, 96, 192, 384, 40, 80, 160, 320]


def ept(n):
    return 12 if n % 3 == 0 else 20 if n % 5 == 0 else 16


# --------------------------------------------------------------- column tiles
def cols_radices(n):
    e, first, m = ept(n), [], n
    if e != 16 and n % e == 0:
        first, m = [e], n // e
    rest = []
    while m > 1:
        rest.append(ct_radix(m, e, 0))
        m //= rest[-1]
    return first + rest


def col_width(n):
    w = 16
    while w > 1 and w * n // ept(n) > 256:
        w >>= 1
    return w


def cols_replay(n, W, inv):
    e, radices = ept(n), cols_radices(n)
    T, ns = W * n // e, 1
    for rad in (radices[::-1] if inv else radices):
        assert e % rad == 0 or rad == 2
        nb, nbl = e // rad, n // rad
        assert nbl * W <= T * nb  # every butterfly has a thread
        reads, writes = set(), set()
        for t in range(T):
            for i in range(nb):
                b = t + i * T
                if b >= nbl * W:
                    continue
                line, j = b % W, b // W
                base = (j // ns) * ns * rad + j % ns
                for r in range(rad):
                    reads.add((j + r * nbl) * W + line)
                    writes.add((base + r * ns) * W + line)
        assert reads == writes == set(range(n * W))
        ns *= rad
    assert ns == n


@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("inv", [False, True])
def test_column_tiles(n, inv):
    for W in (col_width(n), max(32 * ept(n) // n, 2)):  # the box's tiles and a plane's narrow ones
        cols_replay(n, W, inv)


# ----------------------------------------------------------------------- rows
def row_radix(cl, left):
    if cl == 16 and left % 16 == 0:
        return 16
    if cl == 16 and left % 8 == 0:
        return 8
    return 4 if left % 4 == 0 else 2


@pytest.mark.parametrize("n", LENGTHS)
def test_rows(n):
    cl = ept(n)
    tpl = n // cl
    nl, sl = 32 // tpl, n + n // cl
    assert n == cl * tpl and nl * tpl == 32
    at = lambda line, a: line * sl + a + a // cl
    whole = {at(line, a) for line in range(nl) for a in range(n)}
    assert len(whole) == nl * n and max(whole) < nl * sl
    # twiddles w_{ns rad}^{k r} at off + (r - 1) ns + k, as exponents of w_n
    tw, off, ns = {}, 0, cl
    while ns < n:
        rad = row_radix(cl, n // ns)
        for i in range((rad - 1) * ns):
            tw[off + i] = (i % ns) * (i // ns + 1) * (n // (ns * rad))
        off += (rad - 1) * ns
        ns *= rad
    assert off < n
    # first stage: lane (line, j) transforms elements j + r tpl and writes cl neighbouring ones
    writes = [(lane // tpl) * sl + (lane % tpl) * (cl + 1) + r for lane in range(32) for r in range(cl)]
    assert len(set(writes)) == len(writes) and set(writes) == whole
    off, ns = 0, cl
    while ns < n:
        rad = row_radix(cl, n // ns)
        nb, nbl = cl // rad, n // rad
        assert cl % rad == 0 and nbl % cl == 0 and ns % cl == 0
        reads, writes = [], []
        for lane in range(32):
            for i in range(nb):
                b = lane + 32 * i
                line, j = b // nbl, b % nbl
                k, base = j % ns, (j // ns) * ns * rad + j % ns
                for r in range(rad):
                    reads.append(line * sl + j + j // cl + r * (nbl + nbl // cl))
                    assert reads[-1] == at(line, j + r * nbl)
                    writes.append(line * sl + base + base // cl + r * (ns + ns // cl))
                    assert writes[-1] == at(line, base + r * ns)
                    if r:
                        assert tw[off + (r - 1) * ns + k] == k * r * (n // (ns * rad))
        assert set(reads) == set(writes) == whole and len(reads) == len(writes) == nl * n
        off += (rad - 1) * ns
        ns *= rad
    assert ns == n


# ----------------------------------------------------------- FP64 small grids
def fine_radix(left):
    return 4 if left % 4 == 0 else 5 if left % 5 == 0 else 3 if left % 3 == 0 else 2


def fine_threads(n, nl):
    per = n // 3 if n % 3 == 0 else n // 4
    return (max(per * nl, 1) + 31) // 32 * 32


def fine_replay(n, nl, T, cols):
    ll = nl.bit_length() - 1
    sl = n + n // 8 + 1
    at = (lambda line, a: (a << ll) + line) if cols else (lambda line, a: line * sl + a + a // 8)
    whole = {at(line, a) for line in range(nl) for a in range(n)}
    assert len(whole) == nl * n and max(whole) < (n << ll if cols else nl * sl)
    ns = 1
    while ns < n:
        rad = fine_radix(n // ns)
        nbl = n // rad
        B = nbl * nl
        assert B <= 2 * T  # at most two butterflies per thread
        reads, writes = [], []
        for b in range(B):
            line, j = (b & (nl - 1), b >> ll) if cols else (b // nbl, b % nbl)
            k = j % ns
            for r in range(rad):
                reads.append(at(line, j + r * nbl))
                writes.append(at(line, (j // ns) * ns * rad + k + r * ns))
                assert 0 <= k * r * (n // (ns * rad)) < n  # the root's index
        assert set(reads) == set(writes) == whole and len(reads) == len(writes) == nl * n
        ns *= rad
    assert ns == n


def fine_cl(n):
    cl = 3 if n % 3 == 0 else 5 if n % 5 == 0 else 4
    while n // cl > 32:
        cl *= 2
    return cl


@pytest.mark.parametrize("n", LENGTHS)
def test_small_grid_passes(n):
    # density: LP pairs of rows
    lp = max(1, 128 // n)
    assert fine_threads(n, lp) <= 256
    fine_replay(n, lp, fine_threads(n, lp), False)
    # strided: eight columns, halved to one warp where SMs are left without a block
    lw = 3
    while lw > 0 and (n << lw) // 4 > 256:
        lw -= 1
    for k in range(lw + 1):
        assert fine_threads(n, 1 << k) <= 256
        fine_replay(n, 1 << k, fine_threads(n, 1 << k), True)
    # C2R, exponential and solve: tpl lanes per row
    tpl = n // fine_cl(n)
    assert tpl <= 32 and tpl & (tpl - 1) == 0 and fine_cl(n) <= 16
    for rows, phi in ((2, False), (1, False), (1, True)):  # a complex row, a real pair, Phi_d alone
        lp = max(1, 32 // (rows * tpl))
        T = fine_threads(n, lp) if phi else max(rows * lp * tpl, fine_threads(n, lp))
        T = (T + 31) // 32 * 32
        assert T <= 256
        fine_replay(n, lp, T, False)
