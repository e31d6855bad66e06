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
