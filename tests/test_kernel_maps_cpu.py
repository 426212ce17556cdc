"""Host checks of the index maps of the kernels that move whole rows (restated from solver_kernels.cuh): the
tensor-copied z tiles with their swizzled exchange, the y-pass with the lines in registers, the short y
tiles, the rows of the x-stage that arrive by bulk copies, and the tile layouts by type. Every address lies inside its
buffer, every value is touched once, copies are aligned and add up to what their barrier expects, and the
lane programs give the transforms."""

import numpy as np
import pytest

CUBES = (8, 12, 16, 24, 32, 48, 64, 96, 128, 256, 512, 1024)
BOXES = ((32, 16, 24), (24, 48, 16), (1024, 512, 256))
SHAPES = [(n, n, n) for n in CUBES] + list(BOXES)


def pow2_part(n):
    return n & -n


def odd_ld(lines):
    return lines | 1


def padt(p, cb):
    return p + (p >> 3) if cb == 16 else p + (p >> 4)


def padt_len(L, cb):
    return padt(L - 1, cb) + 1 if cb == 16 else L + L // 16 + 1


class ZLay:
    """Tile layout of the FP32 z tiles and the short FP32 y tiles for lines of M values."""

    def __init__(self, M):
        self.M = M
        self.pad = 4 if M in (12, 16) else 8 if M in (24, 32, 64) else 16
        self.res = 4 if M in (12, 16) else 6 if M == 24 else 2 if M in (32, 64) else 11 if M == 48 else -1

    def row(self, p):
        return p + p // self.pad

    @property
    def rows(self):
        return self.row(self.M - 1) + 1

    def ld(self, lines):
        return lines | 1 if self.res < 0 else lines + (self.res - lines % 16 + 16) % 16


def zbytes(M, t, cb):
    if cb == 8:
        z = ZLay(M)
        return z.rows * z.ld(6 * t) * cb
    return padt_len(M, cb) * odd_ld(6 * t) * cb


def ztx(N, M, cb):
    t = min(16, pow2_part(N))
    while t > 1 and zbytes(M, t, cb) > (113 if cb == 16 else 112) * 1024 and not (t * cb <= 32 and zbytes(M, t, cb) <= 200 * 1024):
        t //= 2
    return t


def _widths(N, cb, which):
    import ctypes

    from paper_1602_03638_gb300 import _lib
    from paper_1602_03638_gb300 import build as B

    B.build()
    buf = (ctypes.c_int * 8)()
    n = _lib.lib().dns_tile_widths(N, 0 if cb == 8 else 1, which, buf, 8)
    assert n >= 0, _lib.last_error()
    return list(buf[:n])


# ---------------------------------------------------------------- z tiles of k_zpass

@pytest.mark.parametrize("cb", [8, 16])
@pytest.mark.parametrize("shape", SHAPES)
def test_z_tiles_lie_inside_their_allocation(shape, cb):
    N, _, NZ = shape
    M = NZ // 2
    offered = _widths(N, cb, 1) if shape[0] == shape[1] == shape[2] and N <= 128 else []
    for t in [ztx(N, M, cb)] + offered:
        assert N % t == 0
        assert zbytes(M, t, cb) <= (227 * 1024 if t not in offered else 112 * 1024)
        if cb == 8:
            z = ZLay(M)
            row, ld = z.row, z.ld(6 * t)
        else:
            row, ld = (lambda p: padt(p, 16)), odd_ld(6 * t)
        at = [row(k) * ld + f for k in range(M) for f in range(6 * t)]
        assert ld >= 6 * t and len(set(at)) == len(at) and max(at) * cb < zbytes(M, t, cb)
        if cb == 8 and ld % 2 == 0 and t % 2 == 0:  # pairs of columns by 16-byte copies, on both sides
            assert all((row(k) * ld + f * t) % 2 == 0 for k in range(M) for f in range(6))
            assert N % 2 == 0


# ---------------------------------------------------------------- short FP32 y tiles

def _line_radix0(L, V):
    three = L % 3 == 0
    a = (L // 3 if three else L).bit_length() - 1
    if V == 1:
        return 3 if three else (4 if a >= 2 and not (a == 3) else (8 if a == 3 else 2))
    return 8 if a >= 3 else {1: 2, 2: 4}[a]


@pytest.mark.parametrize("shape", [s for s in SHAPES if s[1] <= 128])
def test_short_y_tiles_read_and_store_their_rows_once(shape):
    N, L, _ = shape
    widths = [min((128 // 8) if inv else 8, pow2_part(N)) for inv in (0, 1)]
    if shape[0] == shape[1] == shape[2]:
        widths += _widths(N, 8, 0)
    z = ZLay(L)
    for tx in set(widths):
        ld, nt = z.ld(tx), min(32 * tx, 128)
        vx = 2 if ld % 2 == 0 and tx % 2 == 0 else 1
        assert N % tx == 0 and z.rows * ld * 8 <= 227 * 1024
        for V in (0, 1):
            nb0 = L // _line_radix0(L, V)
            g = min(1 if nb0 >= 32 else 2 if nb0 >= 16 else 4 if nb0 >= 8 else 8 if nb0 >= 4 else 16, tx // 4 if tx >= 4 else 1)
            cols = [c + i for w in range(nt // 32) for c in range(w * g, tx, nt // 32 * g) for i in range(g)]
            assert sorted(cols) == list(range(tx))
        for kmax3 in sorted({L, L + 2, 3, 3 * (L // 4), 3 * (L // 2)} - {0}):
            R = min((kmax3 - 1) // 3, L // 2 - 1)
            lo, gap = R + 1, 0 if 3 * (L // 2) < kmax3 else L - 2 * R - 1
            inside = {y for y in range(L) if 3 * abs(y if y < L // 2 else y - L) < kmax3}
            for skip in (0, gap):
                seen = {}
                for e in range(tx // vx * (L - skip)):
                    x, r = e % (tx // vx) * vx, e // (tx // vx)
                    y = r if r < lo else r + skip
                    assert 0 <= y < L and (z.row(y) * ld + x) % vx == 0
                    for i in range(vx):
                        assert z.row(y) * ld + x + i < z.rows * ld
                        seen[(y, x + i)] = seen.get((y, x + i), 0) + 1
                assert set(seen.values()) == {1}
                rows = {y for y, _ in seen}
                assert rows == (set(range(L)) if skip == 0 else inside)


# ---------------------------------------------------------------- y-pass with the lines in registers

@pytest.mark.parametrize("NY", [256, 512, 1024])
def test_register_lines_of_the_y_pass_are_the_transform(NY):
    E = 16 if NY == 256 else 32
    T, TX = NY // E, 8 if NY == 1024 else 16
    B, ROW = E // T, T * TX + (8 if TX == 8 else 0)
    assert TX * T == 256
    rng = np.random.default_rng(NY)
    x = rng.standard_normal(NY) + 1j * rng.standard_normal(NY)
    s = {}
    for l in range(T):
        y = [l + T * m for m in range(E)]
        v = np.fft.fft(x[y]) * np.exp(-2j * np.pi * l * np.arange(E) / NY)
        for j in range(E):
            for c in (0, TX - 1):
                a = j * ROW + l * TX + c
                assert 0 <= a < E * ROW and a not in s
                s[a] = v[j]
    out = {}
    for l in range(T):
        for b in range(B):
            w = np.fft.fft([s[(l + T * b) * ROW + q * TX] for q in range(T)])
            for k in range(T):
                assert l + T * b + E * k not in out
                out[l + T * b + E * k] = w[k]
    got = np.array([out[k] for k in range(NY)])
    assert np.abs(got - np.fft.fft(x)).max() < 1e-10
    # the rows read or stored: |ky| < lim; lim = NY: all
    for kmax3 in (NY, NY + 2):
        lim = min((kmax3 + 2) // 3, NY // 2)
        for y in range(NY):
            ky = y if y < NY // 2 else y - NY
            assert (y < lim or y > NY - lim) == (3 * abs(ky) < kmax3)


# ---------------------------------------------------------------- x-stage rows by bulk copies

@pytest.mark.parametrize("N", [128, 256, 512, 1024])
def test_bulk_rows_of_the_x_stage(N):
    ls = padt_len(N, 8)
    wide = ((6 * ls + 1) // 2 * 2 + 9 * N) * 8 <= 64 * 1024
    xst = ((6 if wide else 3) * ls + 1) // 2 * 2
    assert (xst + 9 * N) * 8 <= 100 * 1024 and xst * 8 % 16 == 0 and N * 8 % 16 == 0
    for f in range(3):  # the rows of W: 16-byte aligned, unpadded, each inside its own padded line
        start = (f * ls + 1) // 2 * 2
        assert start * 8 % 16 == 0 and f * ls <= start and start + N <= (f + 1) * ls
    if not wide:  # omega's work lines lie over the rows 3 .. 8
        assert 3 * N + 3 * ls <= 9 * N
    for kmax3 in range(3, 3 * N // 2 + 3):
        R = (kmax3 + 2) // 3 - 1
        lo, hi = (R + 2) // 2 * 2, (N - R) // 2 * 2
        if lo >= hi:
            lo = hi = N
        assert lo * 8 % 16 == 0 and hi * 8 % 16 == 0 and 0 < lo <= hi <= N
        copied = set(range(lo)) | set(range(hi, N))
        assert {j for j in range(N) if 3 * abs(j if j < N // 2 else j - N) < kmax3} <= copied
        copies = [lo * 8] + ([(N - hi) * 8] if hi < N else [])
        assert all(c > 0 and c % 16 == 0 for c in copies) and sum(copies) == (lo + N - hi) * 8


# ---------------------------------------------------------------- tensor-copied z tiles

class ZTma:
    def __init__(self, M):
        self.M = M
        self.TX = 4096 // M
        self.CX = min(self.TX, 16)
        self.ROWB = self.CX * 8
        self.CB, self.FB = M * self.ROWB, 32768
        self.HL = 8 if M == 128 else 16
        self.V = M // self.HL
        self.GL = 32 // self.HL
        self.NW = 24 if self.V == 16 else 12
        self.SH, self.MASK = (0 if self.ROWB == 128 else 1), self.ROWB // 16 - 1

    def at(self, r):
        return r * self.ROWB | ((r >> self.SH) & self.MASK) * 16

    def lane(self, lane):
        h = (lane & 7) | ((lane >> 4) << 3) if self.HL == 16 else lane & 7
        cb = (lane >> 3) & 1
        hp = (self.HL - h) & (self.HL - 1)
        return h, cb, (hp & 7) | (cb << 3) | ((hp >> 3) << 4) if self.HL == 16 else (lane & 24) | hp

    def row(self, lane, l, r):
        _, cb, _ = self.lane(lane)
        x = l + ((lane >> 4) * 2 if self.HL == 8 else 0)
        return x // self.CX * self.CB + r * self.ROWB + (((x % self.CX) // 2) ^ ((r >> self.SH) & self.MASK)) * 16 + cb * 8

    def copied(self, x, k):
        """Where the copies of the hardware's swizzle put column x (of all the fields') at plane k."""
        chunk = ((x % self.CX) // 2) ^ ((k * self.ROWB // 128) % (self.ROWB // 16))
        return x // self.CX * self.CB + k * self.ROWB + chunk * 16 + (x % 2) * 8

    def fft(self, v, la, h, mem):
        """zt_fft for the lanes of a warp: v[lane][m], la[lane]; the twiddles as their formula."""
        M, R = self.M, self.V
        written = set()

        def put(a, x):
            assert a not in written and a % 8 == 0 and 0 <= a < 6 * self.FB
            written.add(a)
            mem[a // 8] = x

        for i in range(32):
            t = np.fft.fft(v[i])
            if M != 256:
                t = t * np.exp(-2j * np.pi * h[i] * np.arange(R) / M)
            for r in range(R):
                put((la[i] + h[i] * R * self.ROWB) ^ self.at(r), t[r])
        out = []
        for i in range(32):
            if M == 256:
                a = np.array([mem[((la[i] ^ self.at(m)) + m * 16 * self.ROWB) // 8] for m in range(16)])
                out.append(np.fft.fft(a * np.exp(-2j * np.pi * h[i] * np.arange(16) / M)))
            else:
                q = [(la[i] ^ self.at(g)) + g * R * self.ROWB for g in range(R // 2)]
                a = np.fft.fft([mem[p // 8] for p in q])
                b = np.fft.fft([mem[(p + R // 2 * self.ROWB) // 8] for p in q])
                w = np.empty(R, complex)
                w[0::2], w[1::2] = a, b
                out.append(w)
        return out, written


@pytest.mark.parametrize("M", [128, 256, 512])
def test_tensor_tile_addresses(M):
    z = ZTma(M)
    assert 3 * (z.TX // z.CX) * z.CB == 3 * z.FB and (6 * z.TX) // z.CX * z.CB == 6 * z.FB
    assert M % min(M, 256) == 0 and z.CX * 8 % 16 == 0  # whole copies, rows of a multiple of 16 bytes
    lines = [w * z.GL + z.GL * z.NW * i for w in range(z.NW) for i in range(3 * z.TX)]
    for f0 in (0, 3):
        cols = []
        for w in range(z.NW):
            for l in range(f0 * z.TX + z.GL * w, (f0 + 3) * z.TX, z.GL * z.NW):
                cols += sorted({l + ((lane >> 4) * 2 if z.HL == 8 else 0) + z.lane(lane)[1] for lane in range(32)})
        assert sorted(cols) == list(range(f0 * z.TX, (f0 + 3) * z.TX))
    assert lines
    # a lane's rows are where the copies put its column, and its other rows at a fixed distance
    for l in (0, z.GL, 3 * z.TX, 6 * z.TX - z.GL):
        for lane in range(32):
            h, cb, partner = z.lane(lane)
            x = l + ((lane >> 4) * 2 if z.HL == 8 else 0) + cb
            for m in range(z.V):
                assert z.row(lane, l, h) + m * z.HL * z.ROWB == z.copied(x, h + z.HL * m)
            assert z.lane(partner)[0] == (z.HL - h) % z.HL and z.lane(partner)[1] == cb and z.lane(partner)[2] == lane


@pytest.mark.parametrize("M", [128, 256, 512])
def test_tensor_tile_transforms(M):
    z = ZTma(M)
    HL, V, STEP = z.HL, z.V, z.HL * z.ROWB
    rng = np.random.default_rng(M)
    l = 3 * z.TX + z.GL  # some lines of omega
    mem = np.full(6 * z.FB // 8, np.nan, complex)
    X = rng.standard_normal((6 * z.TX, M)) + 1j * rng.standard_normal((6 * z.TX, M))
    lanes = [z.lane(i) for i in range(32)]
    h, cb, partner = zip(*lanes)
    cols = [l + ((i >> 4) * 2 if HL == 8 else 0) + cb[i] for i in range(32)]
    for x in set(cols):
        for k in range(M):
            mem[z.copied(x, k) // 8] = X[x, k]
    own = {z.copied(x, k) for x in set(cols) for k in range(M)}
    ld = lambda a: mem[a // 8]
    wk = lambda i, m: np.exp(-2j * np.pi * (h[i] + HL * m) / (2 * M))
    # c2r
    pa = [z.row(i, l, h[i]) for i in range(32)]
    pb = [z.row(i, l, HL - h[i]) for i in range(32)]
    v = np.empty((32, V), complex)
    zq = np.empty((32, V // 2), complex)
    for i in range(32):
        for m in range(V // 2):
            if m == 0:
                y = ld(pa[i] + V // 2 * STEP) if h[i] == 0 else ld(pb[i] + (V - 1) * STEP)
                xk, xm, w1 = (y, y, -1j) if h[i] == 0 else (ld(pa[i]), y, wk(i, 0))
            else:
                xk, xm, w1 = ld(pa[i] + m * STEP), ld(pb[i] + (V - 1 - m) * STEP), wk(i, m)
            A, Bv = xk + np.conj(xm), xk - np.conj(xm)
            P = 1j * np.conj(w1) * Bv
            v[i, m], zq[i, m] = np.conj(A + P), A - P
    for i in range(32):
        for q in range(V // 2, V):
            v[i, q] = zq[partner[i], V - 1 - q]
    for i in range(32):
        if h[i] == 0:
            x0 = ld(pa[i])
            v[i, V // 2] = v[i, 0]
            for q in range(V // 2 + 1, V):
                v[i, q] = zq[i, V - q]
            v[i, 0] = x0.real * (1 - 1j)
    v, written = z.fft(v, pa, h, mem)
    assert written == own  # the exchange stays inside the lines of the warp
    for i in range(32):
        for m in range(V):
            mem[(pa[i] + m * STEP) // 8] = np.conj(v[i][m])
    for x in set(cols):
        half = np.concatenate([X[x], [0]])
        half[0] = half[0].real
        ref = np.fft.irfft(half, 2 * M) * 2 * M
        got = np.array([mem[z.copied(x, n) // 8] for n in range(M)])
        assert np.abs(got - (ref[0::2] + 1j * ref[1::2])).max() < 1e-9
    # r2c of the same lines
    phys = {x: np.array([mem[z.copied(x, n) // 8] for n in range(M)]) for x in set(cols)}
    v = [np.array([ld(pa[i] + m * STEP) for m in range(V)]) for i in range(32)]
    v, written = z.fft(v, pa, h, mem)
    assert written == own
    for i in range(32):
        line = np.empty(2 * M)
        line[0::2], line[1::2] = phys[cols[i]].real, phys[cols[i]].imag
        ref = np.fft.rfft(line)
        for m in range(V):
            zo = v[i][(V - m) % V] if h[i] == 0 else v[partner[i]][V - 1 - m]
            A, Bv = v[i][m] + np.conj(zo), v[i][m] - np.conj(zo)
            assert abs(0.5 * (A - 1j * wk(i, m) * Bv) - ref[h[i] + HL * m]) < 1e-8
