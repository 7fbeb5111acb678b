"""Rounding of the stencils, at fields where it can be told apart exactly."""
import numpy as np
import pytest

from oracle import dirac
from paper_1211_0126_gb300 import synthetic as S
from paper_1211_0126_gb300 import tsm

pytestmark = pytest.mark.gpu


def _unit_gauge(dims):
    U = np.zeros(S.gauge_field(dims, 0.3, 1).shape, dtype=np.complex128)
    U[...] = np.eye(3)
    return U


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (12, 12, 12, 12)])
@pytest.mark.parametrize("mu", [0, 1, 2, 3])
@pytest.mark.parametrize("dagger", [False, True])
def test_fp64_hops_of_a_direction_round_once(ctx, dims, mu, dagger):
    """Unit links, one component 1 at x + mu and 2^-53 at x - mu: the lower
    components of site x are their difference times a unit, 1 - 2^-53, which FP64
    holds exactly; formed as 2 * 1 - (1 + 2^-53) it would be 1.  kappa = 1 and mu
    = 0, so that D applies H without another rounding (both FP64 kernels of D)."""
    U = _unit_gauge(dims)
    ctx.load_gauge(U, dims, 1.0, 0.0, antiperiodic_t=False)
    a = np.zeros(S.random_spinor(dims, 1).shape, dtype=np.complex128)
    b = np.zeros_like(a)
    x = [2, 2, 2, 2]
    for f, step, value in ((a, 1, 1.0), (b, -1, 2.0 ** -53)):
        y = list(x)
        y[mu] += step
        f[y[3], y[2], y[1], y[0], 0, 1] = value
    hops = [dirac.hop(U, f, dims, antiperiodic_t=False, adjoint=dagger) for f in (a, b)]
    want = (a + b) - (hops[0] + hops[1])   # every sum has at most two terms: one rounding
    assert np.any(np.abs(want) == 1 - 2.0 ** -53)
    got = ctx.dslash(a + b, tsm.TM_OP_FULL, dagger, tsm.TSM_F64)
    assert np.array_equal(got, want)


def _dyadic_gauge(dims, factors, seed):
    """SU(3) links exact in binary: products of (+-1 +- i +- j +- k) / 2 in the
    three SU(2) subgroups, entries multiples of 2^-factors."""
    rng = np.random.default_rng(seed)
    shape = S.gauge_field(dims, 0.3, 1).shape[:-2]
    U = np.zeros(shape + (3, 3), dtype=np.complex128)
    U[...] = np.eye(3)
    for n in range(factors):
        i, j = ((0, 1), (1, 2), (0, 2))[n % 3]
        a = rng.choice([-0.5, 0.5], shape + (4,))
        g = np.zeros_like(U)
        g[...] = np.eye(3)
        g[..., i, i], g[..., i, j] = a[..., 0] + 1j * a[..., 1], a[..., 2] + 1j * a[..., 3]
        g[..., j, i], g[..., j, j] = -a[..., 2] + 1j * a[..., 3], a[..., 0] - 1j * a[..., 1]
        U = U @ g
    return U


def _hop_of_products(U, psi, real, wide):
    """H psi in arithmetic `real` (complex as two arrays), every SU(3) product as
    the sum of three complex products, each part a multiplication and a
    multiply-add (exact in `wide`, rounded once).  FP32 links: two rows rounded, the
    third formed from them."""
    def fma(a, b, c):
        return (wide(a) * wide(b) + wide(c)).astype(real)

    def times(a, b):                      # a b
        return (fma(a[0], b[0], -(a[1] * b[1])), fma(a[0], b[1], a[1] * b[0]))

    def add(a, b, s=1):
        return (a[0] + s * b[0], a[1] + s * b[1])

    def unit(a, k):                       # i^k a
        return [a, (-a[1], a[0]), (-a[0], -a[1]), (a[1], -a[0])][k % 4]

    U = (U.real.astype(real), U.imag.astype(real))
    if real == np.float32:
        r = [[(U[0][..., a, b], U[1][..., a, b]) for b in range(3)] for a in range(2)]
        w = [add(times(r[0][(c + 1) % 3], r[1][(c + 2) % 3]), times(r[0][(c + 2) % 3], r[1][(c + 1) % 3]), -1)
             for c in range(3)]
        for c in range(3):
            U[0][..., 2, c], U[1][..., 2, c] = w[c][0], -w[c][1]
    v = [(psi.real[..., s, :].astype(real), psi.imag[..., s, :].astype(real)) for s in range(4)]
    # of spin s the projected spins p = 0, 1 take spin q times i^k (1 + gamma_mu), and spin q of the result takes
    # h_p times i^-k; the opposite projector has the opposite sign
    pair = {0: ((3, 3), (2, 3)), 1: ((3, 2), (2, 0)), 2: ((2, 3), (3, 1)), 3: ((2, 0), (3, 0))}
    acc = [(np.zeros_like(v[0][0]), np.zeros_like(v[0][0])) for _ in range(4)]
    for mu in range(4):
        for forward in (True, False):
            s = -1 if forward else 1
            ax = {0: -2, 1: -3, 2: -4, 3: -5}[mu]
            w = [tuple(np.roll(x, -1 if forward else 1, axis=ax) for x in y) for y in v]
            ur, ui = U[0][..., mu, :, :], U[1][..., mu, :, :]
            if not forward:
                ur, ui = [np.swapaxes(np.roll(x, 1, axis={0: 3, 1: 2, 2: 1, 3: 0}[mu]), -1, -2) for x in (ur, -ui)]
            for p in range(2):
                q, k = pair[mu][p]
                h = add(w[p], unit(w[q], k), s)
                rows = []
                for a in range(3):
                    t = [times((ur[..., a, b], ui[..., a, b]), (h[0][..., b], h[1][..., b])) for b in range(3)]
                    rows.append(add(add(t[0], t[1]), t[2]))
                g = tuple(np.stack([r[c] for r in rows], -1) for c in range(2))
                acc[p] = add(acc[p], g)
                acc[q] = add(acc[q], unit(g, -k), s)
    return np.stack([np.stack(a, -1) for a in acc], -3)   # [..., spin, colour, re / im]


@pytest.mark.parametrize("links", ["random", "near the identity"])
@pytest.mark.parametrize("prec,dims", [(tsm.TSM_F32, (12, 12, 12, 12)), (tsm.TSM_F64, (8, 8, 8, 8))])
def test_hop_error_no_larger_than_that_of_summed_products(ctx, prec, dims, links):
    """Rounding error of H psi against 64 (FP64: extended) bits, on fields that the
    tier holds exactly; random links are exact too, so that only the sums round.
    Yardstick: the same error of sums of separately formed products, in numpy.  N
    independent errors on each side: the ratio of their rms values scatters by
    1 / sqrt(N); three times that is allowed."""
    real, wide = (np.float32, np.float64) if prec == tsm.TSM_F32 else (np.float64, np.longdouble)
    U = _dyadic_gauge(dims, 7, 3) if links == "random" else S.gauge_field(dims, 0.25, 3)
    ctx.load_gauge(U, dims, 0.1, 0.0, antiperiodic_t=False)
    psi = S.random_spinor(dims, 4) * dirac.odd_mask(dims)
    psi = psi.real.astype(real).astype(np.float64) + 1j * psi.imag.astype(real).astype(np.float64)
    even = np.broadcast_to(dirac.even_mask(dims), psi.shape) != 0
    exact = _hop_of_products(U, psi, wide, wide)[even]
    rounded = _hop_of_products(U, psi, real, wide)[even]
    got = ctx.dslash(psi, tsm.TM_OP_HOP_EO, False, prec)
    got = np.stack([got.real, got.imag], -1)[even]
    rms = [float(np.sqrt(np.mean((x.astype(wide) - exact) ** 2))) for x in (got, rounded)]
    print("rms error: kernel %.5e, sums of products %.5e, ratio %.5f" % (rms[0], rms[1], rms[0] / rms[1]))
    assert rms[0] <= rms[1] * (1 + 3 / np.sqrt(exact.size))
