"""The complex64 hybrid cycle restated in numpy with every FP32 rounding in its place, for
tests that compare bits: which products are fused into an addition, and the order of the
sums.  Complex vectors are pairs (real part, imaginary part) of float32 arrays."""
import numpy as np

f32 = np.float32


def pair(z):
    z = np.asarray(z)
    return z.real.astype(f32), z.imag.astype(f32)


def fma(a, b, c):
    """a b + c rounded once (the product of two FP32 numbers is exact in FP64; the sum is
    rounded there first, which matters for one value in 2^29)."""
    return (np.asarray(a, np.float64) * np.asarray(b, np.float64) + np.asarray(c, np.float64)).astype(f32)


def cmul(a, b, turned=False):
    """a b: the product with a's real part is fused into the sum, with `turned` the one with
    a's imaginary part in the imaginary part of the result."""
    re = fma(a[0], b[0], -(a[1] * b[1]))
    return re, fma(a[1], b[0], a[0] * b[1]) if turned else fma(a[0], b[1], a[1] * b[0])


class Op32:
    """The complex64 operator on an n^dim grid: mask, absorbing layer or stored k^2."""

    def __init__(self, dim, n, k0, mask, cells, strength=0.5, k2=None):
        self.dim, self.n, self.shape = dim, n, (n,) * dim
        self.fluid = np.asarray(mask).reshape(-1) == 0
        ax = np.meshgrid(*[np.arange(n)] * dim, indexing="ij")
        self.colour = (sum(ax) % 2).reshape(-1)
        h = 1.0 / (n - 1)
        hinv2 = 1.0 / (h * h)
        self.hinv2 = f32(hinv2)
        if k2 is None:
            m = np.maximum(0, cells - np.stack([np.minimum(a, n - 1 - a) for a in ax]).reshape(dim, -1)).max(0)
            im = k0 * k0 * ((strength * (m / cells)) * (m / cells))
            re = np.full(n ** dim, k0 * k0 - 2.0 * dim / (h * h))
            self.diag = re.astype(f32), im.astype(f32)
        else:
            k2 = np.asarray(k2).reshape(-1)
            re, im = k2.real - 2.0 * dim * hinv2, k2.imag
            self.diag = k2.real.astype(f32) - f32(2 * dim) * self.hinv2, im.astype(f32)
        d2 = re * re + im * im
        self.invd = (re / d2).astype(f32), (-im / d2).astype(f32)

    def conj(self, v, conj):
        return (v[0], -v[1]) if conj else v

    def neighbours(self, x, axis):
        """the two neighbour values along an axis (zero where they are masked or do not exist)"""
        p = np.pad(np.where(self.fluid, x, f32(0)).reshape(self.shape), 1)
        cut = lambda s: p[tuple(slice(1 + s, self.n + 1 + s) if q == axis else slice(1, self.n + 1)  # noqa: E731
                                for q in range(self.dim))].reshape(-1)
        return cut(-1), cut(1)

    def nbr_sum(self, x):
        """pairs along x, y and z, then (x + y) + z"""
        s = [np.add(*self.neighbours(x, a)) for a in range(self.dim - 1, -1, -1)]
        return s[0] + s[1] if self.dim == 2 else (s[0] + s[1]) + s[2]

    def rhs_minus_nbrs(self, f, x):
        return tuple(fma(-self.hinv2, self.nbr_sum(q), p) for p, q in zip(f, x))

    def sweeps(self, kind, omega, count, f, x=None, conj=False):
        """red-black Gauss-Seidel, SOR or SSOR sweeps, in place of x or (x None) from zero"""
        om = f32(1.0 if kind == "rbgs" else omega)
        invd = self.conj(self.invd, conj)
        zero = x is None                                   # only the first half-sweep reads nothing
        x = tuple(np.zeros_like(p) for p in f) if zero else x
        for _ in range(count):
            for c in (0, 1, 1, 0) if kind == "ssor" else (0, 1):
                v = cmul(invd, f, turned=True) if zero else cmul(invd, self.rhs_minus_nbrs(f, x))
                v = tuple(np.where(self.fluid, p, q) for p, q in zip(v, f))
                if om != 1:
                    v = tuple(om * p for p in v) if zero else tuple(fma(om, p - q, q) for p, q in zip(v, x))
                x = tuple(np.where(self.colour == c, p, q) for p, q in zip(v, x))
                zero = False
        return x

    def jacobi(self, omega, count, f, x=None, conj=False):
        """damped-Jacobi sweeps: (1 - omega) x + omega D^-1 (f - h^-2 sum of neighbours)"""
        om = f32(omega)
        w1 = f32(1) - om
        invd = self.conj(self.invd, conj)
        x = tuple(np.zeros_like(p) for p in f) if x is None else x
        for _ in range(count):
            v = cmul(invd, self.rhs_minus_nbrs(f, x))
            x = tuple(np.where(self.fluid, fma(w1, q, om * p), fma(om, g - q, q)) for p, q, g in zip(v, x, f))
        return x

    def residual(self, v, z, conj=False):
        """v - A z on fluid nodes, 0 on masked ones; neighbours added one after the other"""
        dz = cmul(self.conj(self.diag, conj), z, turned=True)
        out = []
        for vv, zz, p in zip(v, z, dz):
            s = np.zeros_like(zz)
            for a in range(self.dim - 1, -1, -1):
                for q in self.neighbours(zz, a):
                    s = s + q
            out.append(np.where(self.fluid, vv - fma(self.hinv2, s, p), f32(0)))
        return tuple(out)

    def red_rows(self):
        """the red node of each pair (2m, 2m + 1); N where the last pair has none"""
        m2 = 2 * np.arange((self.fluid.size + 1) // 2)
        return m2 + self.colour[m2]

    def cycle(self, Q, Ainv, v, z, red, conj=False):
        """z + Q A_c^-1 Q^T (v - A z) (z None: no sweeps), the residual on the red rows alone
        (`red`) or on all; Q: the BF16 basis, node-major"""
        r = tuple(np.where(self.fluid, p, f32(0)) for p in v) if z is None else self.residual(v, z, conj)
        z = tuple(np.zeros_like(p) for p in v) if z is None else z
        Q = np.asarray(Q, f32)
        if red:
            rows = np.append(np.arange(self.fluid.size), 0)[self.red_rows()]
            here = (self.red_rows() < self.fluid.size)
            c = [coarse_sum(red_parts(np.where(here[:, None], Q[rows], f32(0)), np.where(here, p[rows], f32(0)))) for p in r]
        else:
            c = [coarse_sum(all_parts(Q, p)) for p in r]
        y = (Ainv.conj() if conj else Ainv) @ (c[0].astype(np.float64) + 1j * c[1].astype(np.float64))
        out = []
        for p, q in zip(z, pair(y)):
            a = np.zeros_like(p)
            for j in range(Q.shape[1]):
                a = fma(Q[:, j], q[j], a)
            out.append(p + a)
        return tuple(out)


def butterfly(v):
    """the 32 lanes (first axis) added pairwise at distances 16, 8, 4, 2, 1"""
    for o in (16, 8, 4, 2, 1):
        v = v + v[np.arange(32) ^ o]
    return v[0]


def chain(q, r):
    """sum of q r along the first axis, one fused multiply-add after the other"""
    a = np.zeros(np.broadcast(q[0], r[0]).shape, f32)
    for p, x in zip(q, r):
        a = fma(p, x, a)
    return a


def red_parts(Q, r):
    """Q^T r of red rows: 8 rows a lane, 256 a warp, tiles 8 blocks apart added in order, the
    block's eight warps in order"""
    M, k = Q.shape
    tiles = -(-M // 256)
    blocks = min(608, -(-tiles // 8))
    q, x = np.zeros((tiles * 256, k), f32), np.zeros(tiles * 256, f32)
    q[:M], x[:M] = Q, r
    t = butterfly(chain(q.reshape(tiles, 32, 8, k).transpose(2, 1, 0, 3), x.reshape(tiles, 32, 8, 1).transpose(2, 1, 0, 3)))
    part = np.zeros((blocks, k), f32)
    for b in range(blocks):
        for w in range(8):
            acc = np.zeros(k, f32)
            for i in range(8 * b + w, tiles, 8 * blocks):
                acc = acc + t[i]
            part[b] = part[b] + acc
    return part


def all_parts(Q, r):
    """Q^T r of all rows: equal shares of the rows, every 32nd row of one in a lane's chain"""
    N, k = Q.shape
    blocks = min(304, max(1, -(-N // 256)))
    share = -(-N // blocks)
    m = -(-share // 32)
    part = np.zeros((blocks, k), f32)
    for b in range(blocks):
        q, x = np.zeros((m * 32, k), f32), np.zeros(m * 32, f32)
        rows = slice(min(N, b * share), min(N, (b + 1) * share))
        q[:rows.stop - rows.start], x[:rows.stop - rows.start] = Q[rows], r[rows]
        part[b] = butterfly(chain(q.reshape(m, 32, k), x.reshape(m, 32, 1)))
    return part


def coarse_sum(part):
    """the partial rows: every 256th in a thread, a butterfly a warp, the eight warps in order"""
    v = np.zeros((256, part.shape[1]), f32)
    for b in range(part.shape[0]):
        v[b % 256] = v[b % 256] + part[b]
    s = np.zeros(part.shape[1], f32)
    for w in range(8):
        s = s + butterfly(v[32 * w:32 * w + 32])
    return s
