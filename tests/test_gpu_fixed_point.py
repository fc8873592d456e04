"""FP64 products in fixed point (csrc/fix.h: FP16 tensor-core slices with 64-bit sums; and
csrc/k_fix_band.cu: integer multiply-adds) at the edges of their tiles and of the range they take.

Bounds, relative to the largest entry: 1e-12 for P_0^-1, the bound of test_base_preconditioner (six
chained contractions, each within a few ulp of its largest product), and 1e-13 for K, that of
test_operator_applies.
"""
import numpy as np
import pytest
import torch

from paper_2311_06926_gb300 import Stokes, synthetic

from gpu_common import dev, host, oracle, relerr
from oracle.matfree import kron3_apply

pytestmark = pytest.mark.gpu


def _ctx(n, p, **kw):
    return Stokes(n, p, max_order=2, max_steps=0, **kw)


# halves of 12 (FMA chains), 13, 16, 17, 32, 33, 41 terms (tiles of 8 outputs, steps of 16 terms, the
# level sums moved every 2 and 5 steps); b = 63 and below, 64, 65, 82: the dense inverse and the line
# solves
@pytest.mark.parametrize("n,p", [(23, 1), (24, 1), (31, 1), (31, 2), (61, 2), (63, 1), (62, 3),
                                 (78, 4)])
def test_base_preconditioner_tile_edges(n, p):
    S, base, _, _ = oracle(n, p)
    x = synthetic.random_vector(S.size, 40 + n)
    ref = np.concatenate([base.pv0_inv(x[:S.n_vel]), base.pq0_inv(x[S.n_vel:])])
    G = _ctx(n, p, autotune=False)
    for fused in (0, 1, 4):
        G.set_tuning(128, 256, fused)
        got = host(G.apply_P(dev(x)))
        assert relerr(got[:S.n_vel], ref[:S.n_vel]) < 1e-12
        assert relerr(got[S.n_vel:], ref[S.n_vel:]) < 1e-12
    G.close()


@pytest.mark.parametrize("n,p", [(29, 2), (63, 1)])
@pytest.mark.parametrize("fused", [0, 1])
def test_lines_outside_the_scaled_range(n, p, fused):
    """Vectors whose lines are too small or too large to be scaled take FMA chains: the result
    scales with the input."""
    G = _ctx(n, p, autotune=False)
    G.set_tuning(256, 256, fused)
    x = dev(synthetic.random_vector(G.size, 3))
    y = host(G.apply_P(x))
    for e in (-900, 800):
        z = host(G.apply_P(x * 2.0 ** e))
        assert relerr(np.ldexp(z, -e), y) < 1e-12
    assert not host(G.apply_P(torch.zeros_like(x))).any()
    G.close()


@pytest.mark.parametrize("n,p", [(29, 2), (63, 1)])
@pytest.mark.parametrize("fused", [0, 1])
@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_nonfinite_entry_reaches_its_whole_tensor_only(n, p, fused, bad):
    """P_0^-1 mixes every entry of a component (or of the pressure) and nothing else."""
    G = _ctx(n, p, autotune=False)
    G.set_tuning(256, 256, fused)
    x = dev(synthetic.random_vector(G.size, 4))
    y = host(G.apply_P(x))
    m = G.n_vel // 3
    for part in range(4):
        lo, hi = part * m, (part + 1) * m if part < 3 else G.size
        xb = x.clone()
        xb[lo + (hi - lo) // 3] = bad
        z = host(G.apply_P(xb))
        assert not np.isfinite(z[lo:hi]).any()
        keep = np.ones(G.size, bool)
        keep[lo:hi] = False
        assert np.array_equal(z[keep], y[keep])
    G.close()


@pytest.mark.parametrize("n,p", [(63, 1), (62, 2), (64, 3), (61, 4)])
def test_pressure_entries_keep_their_own_accuracy(n, p):
    """The pressure block of long lines entry by entry, on vectors of wide range. To first order an
    error of c 2^-53 |M| in M-check, in every direction, moves an entry by c 2^-53 of the sums below.
    c = 40: 16 for the quadrature roundings in which two M-checks differ, 3 (p + 2) for a banded
    Cholesky solve (M-check is totally positive, so |L| |L^T| = M)."""
    S, _, _, _ = oracle(n, p)
    G = _ctx(n, p, autotune=False)
    x = _wide_vector(G, n)
    x[:G.n_vel] = 0.0
    M = S.uv.Mc.astype(np.longdouble)
    inv = np.linalg.inv(S.uv.Mc).astype(np.longdouble)
    for _ in range(3):   # Newton steps in extended precision
        inv = inv + inv @ (np.eye(G.b, dtype=np.longdouble) - M @ inv)
    q = x[G.n_vel:].reshape(G.b, G.b, G.b)

    def passes(D, t):   # D[d] along direction d, in extended precision
        for axis, d in zip((2, 1, 0), D):
            t = np.moveaxis(np.tensordot(t, d, axes=([axis], [1])), -1, axis)
        return t

    ref = 2.0 * passes([inv] * 3, q.astype(np.longdouble))
    a = np.abs(inv).astype(float)
    wide = a @ np.abs(S.uv.Mc) @ a
    size = sum(2.0 * passes([wide if k == d else a for k in range(3)], np.abs(q)) for d in range(3))
    got = host(G.apply_P(dev(x)))[G.n_vel:].reshape(ref.shape)
    G.close()
    assert (np.abs(got - ref) / size).max() < 40 * 2.0 ** -53


# extents from the smallest that takes the fixed-point passes, ragged and whole segments of 8 rows,
# half widths 2 to 6, and 7, which does not (p = 6)
@pytest.mark.parametrize("n,p,nu", [(38, 1, 1.0), (39, 1, 0.3), (38, 2, 2.0), (46, 2, 1.0),
                                    (45, 3, 0.7), (44, 4, 1.0), (43, 5, 3.0), (41, 6, 1.0)])
def test_operator_segment_edges(n, p, nu):
    S, _, Kop, F = oracle(n, p, nu)
    x = synthetic.random_vector(S.size, 60 + n + p)
    G = Stokes(n, p, nu=nu, max_order=2, max_steps=0, autotune=False)
    ref = Kop(x)
    for block in (128, 256, 512):
        G.set_tuning(512, block, 0)
        assert relerr(host(G.apply_K(dev(x))), ref) < 1e-13
    assert relerr(host(G.apply_A(dev(x[:S.n_vel]))), F.apply_A(x[:S.n_vel])) < 1e-13
    G.close()


def test_operator_windows_outside_the_scaled_range():
    """Windows that cannot be scaled take FMA chains: the result scales with the input, a zero
    vector gives zeros, and an infinite or NaN entry reaches the entries that read it only."""
    G = _ctx(41, 3, autotune=False)
    x = dev(synthetic.random_vector(G.size, 5))
    y = host(G.apply_K(x))
    for e in (-900, 800):
        assert relerr(np.ldexp(host(G.apply_K(x * 2.0 ** e)), -e), y) < 1e-13
    assert not host(G.apply_K(torch.zeros_like(x))).any()
    a, b = G.a, G.b
    for bad in (float("inf"), float("nan")):
        xb = x.clone()
        # entry (20, 20, 20) of u1: its products reach 2 (p + 1) = 8 entries along each direction;
        # entries that share a window with it are formed by chains (the same to rounding)
        xb[20 + a * (20 + b * 20)] = bad
        z = host(G.apply_K(xb))
        u1 = np.isfinite(z[:a * b * b].reshape(b, b, a))
        assert not u1[20, 20, 20]
        far = np.ones((b, b, a), bool)
        far[12:29, 12:29, 12:29] = False
        assert u1[far].all()
        assert relerr(z[:a * b * b].reshape(b, b, a)[far], y[:a * b * b].reshape(b, b, a)[far]) < 1e-13
    G.close()


# points per direction below, at and above 48 (where the fixed-point passes begin; p + 2 points per
# element), windows of 8 that hold p = 1..6, and the last segment of 8 rows ragged and whole
@pytest.mark.parametrize("n,p,nu", [(15, 1, 1.0), (16, 1, 0.6), (21, 1, 1.0), (11, 2, 1.0),
                                    (12, 2, 2.0), (10, 3, 1.0), (13, 3, 1.0), (8, 4, 0.5),
                                    (7, 5, 1.0), (10, 5, 1.0), (6, 6, 1.0), (9, 6, 1.0)])
def test_quadrature_segment_edges(n, p, nu):
    """Bound: that of test_quadrature_operator_equals_kronecker_and_oracle."""
    S, _, Kop, F = oracle(n, p, nu)
    x = synthetic.random_vector(S.size, 80 + n + p)
    ref = Kop(x)
    G = Stokes(n, p, nu=nu, max_order=2, max_steps=0, autotune=False, forward="quadrature")
    for block in (128, 256, 512):
        G.set_tuning(512, block, 0)
        assert relerr(host(G.apply_K(dev(x))), ref) < 1e-12
    for e in (-900, 800):   # windows that cannot be scaled take chains
        assert relerr(np.ldexp(host(G.apply_K(dev(x) * 2.0 ** e)), -e), ref) < 1e-12
    G.close()


def _wide_vector(G, seed):
    """Entries of wide range next to each other: steps of 2^-20 along x1, a fall by 4 per entry along
    x2 (12 entries, then again), single entries 1e6 times their neighbours."""
    rng = np.random.default_rng(seed)
    a, b = G.a, G.b
    out = []
    for e1, e2, e3 in ((a, b, b), (b, a, b), (b, b, a), (b, b, b)):
        t = rng.standard_normal((e3, e2, e1))
        t *= np.where(np.arange(e1) // 5 % 2, 1.0, 2.0 ** -20)
        t *= (4.0 ** -(np.arange(e2) % 12))[:, None]
        spikes = rng.integers(0, t.size, 200)
        t.reshape(-1)[spikes] *= 1e6
        out.append(t.reshape(-1))
    return np.concatenate(out)


@pytest.mark.parametrize("n,p,nu", [(60, 1, 1.0), (52, 2, 0.3), (51, 3, 2.0), (49, 4, 1.0),
                                    (47, 5, 1.0)])
def test_operator_entries_keep_their_own_accuracy(n, p, nu):
    """K x entry by entry against the FMA chains, which the same vector times 2^900 takes: each path
    rounds an entry at most once per term of its passes (six sums of at most 2 p + 3 terms, and the
    divergence), relative to the sum of the magnitudes of the entry's own products."""
    S, _, _, _ = oracle(n, p, nu)
    G = Stokes(n, p, nu=nu, max_order=2, max_steps=0, autotune=False)
    x = _wide_vector(G, n)
    m, k, nv = S.uv, kron3_apply, G.n_vel
    M, K, Mc, Tc = (np.abs(t) for t in (m.M, m.K, m.Mc, m.Tc))
    sizes = [(G.b, G.b, G.a), (G.b, G.a, G.b), (G.a, G.b, G.b)]
    u = [np.abs(t).reshape(s) for t, s in zip(np.split(x[:nv], 3), sizes)]
    q = np.abs(x[nv:]).reshape(G.b, G.b, G.b)
    delta = sum(np.pad(t, [(0, 1) if d == ax else (0, 0) for d in range(3)])
                + np.pad(t, [(1, 0) if d == ax else (0, 0) for d in range(3)])
                for t, ax in zip(u, (2, 1, 0)))
    g = k(Mc, Mc, Mc, nu * delta + q)
    size = []
    for c, t in enumerate(u):
        own, other = (K, M), (Mc, Tc)
        A = 0
        for at in range(3):   # the direction that carries K (own) or T-check (another one)
            D = []
            for d in range(3):
                pair = own if d == c else other
                hit = d == at
                D.append(pair[0] if (hit == (d == c)) else pair[1])
            A = A + (2 if at != c else 1) * nu * k(D[2], D[1], D[0], t)
        ax = 2 - c
        size.append((A + g[tuple(slice(0, -1) if d == ax else slice(None) for d in range(3))]
                     + g[tuple(slice(1, None) if d == ax else slice(None) for d in range(3))])
                    .reshape(-1))
    size = np.concatenate(size + [k(Mc, Mc, Mc, delta).reshape(-1)])
    bound = 2.0 * (6 * (2 * p + 3) + 16) * 2.0 ** -53
    for block in (128, 256):
        G.set_tuning(512, block, 0)
        y = host(G.apply_K(dev(x)))
        z = np.ldexp(host(G.apply_K(dev(np.ldexp(x, 900)))), -900)
        assert (np.abs(y - z) / size).max() < bound
    G.close()


# the smallest extents of the fixed-point passes (p = 1: b = 56, else 48) and the largest below, ragged
# and whole segments, half widths 2 to 6, and 7, which does not take them
@pytest.mark.parametrize("n,p,nu", [(54, 1, 1.0), (55, 1, 0.3), (45, 2, 1.0), (46, 2, 2.0),
                                    (49, 3, 0.7), (44, 4, 1.0), (43, 5, 3.0), (46, 6, 1.0)])
def test_operator_at_the_line_of_the_fixed_point_passes(n, p, nu):
    """Bound: that of test_operator_segment_edges; windows that cannot be scaled agree to it."""
    S, _, Kop, F = oracle(n, p, nu)
    x = synthetic.random_vector(S.size, 90 + n + p)
    G = Stokes(n, p, nu=nu, max_order=2, max_steps=0, autotune=False)
    ref = Kop(x)
    for block in (128, 256, 512):
        G.set_tuning(512, block, 0)
        y = host(G.apply_K(dev(x)))
        assert relerr(y, ref) < 1e-13
        for e in (-900, 800):
            assert relerr(np.ldexp(host(G.apply_K(dev(x) * 2.0 ** e)), -e), y) < 1e-13
    assert not host(G.apply_K(torch.zeros(G.size, dtype=torch.float64, device="cuda"))).any()
    assert relerr(host(G.apply_A(dev(x[:S.n_vel]))), F.apply_A(x[:S.n_vel])) < 1e-13
    G.close()


# several items: the smallest extents of the fixed-point passes, and below
@pytest.mark.parametrize("n,p,nrhs", [(39, 1, 2), (46, 2, 6), (45, 3, 3), (44, 4, 2)])
def test_operator_of_several_items(n, p, nrhs):
    """Bound: that of test_operator_segment_edges, item by item."""
    S, _, Kop, _ = oracle(n, p)
    G = Stokes(n, p, max_order=2, max_steps=1, precision="tf32", nrhs=nrhs, autotune=False)
    X = [synthetic.random_vector(S.size, 200 + n + k) for k in range(nrhs)]
    for block in (128, 256):
        G.set_tuning(512, block, 0)
        got = np.split(host(G.apply_K(dev(np.concatenate(X)))), nrhs)
        for x, y in zip(X, got):
            assert relerr(y, Kop(x)) < 1e-13
    G.close()


# points per direction from 72 on (p + 2 per element), where the fixed-point evaluation passes begin,
# and the largest below; the last segment of 8 rows ragged and whole
@pytest.mark.parametrize("n,p,nu", [(23, 1, 1.0), (24, 1, 0.6), (25, 1, 1.0), (18, 2, 2.0),
                                    (19, 2, 1.0), (15, 3, 1.0), (12, 4, 0.5), (13, 4, 1.0),
                                    (11, 5, 1.0), (9, 6, 1.0), (10, 6, 1.0)])
def test_quadrature_at_the_line_of_the_fixed_point_passes(n, p, nu):
    """Bound: that of test_quadrature_operator_equals_kronecker_and_oracle."""
    S, _, Kop, F = oracle(n, p, nu)
    x = synthetic.random_vector(S.size, 80 + n + p)
    ref = Kop(x)
    G = Stokes(n, p, nu=nu, max_order=2, max_steps=0, autotune=False, forward="quadrature")
    for block in (128, 256, 512):
        G.set_tuning(512, block, 0)
        assert relerr(host(G.apply_K(dev(x))), ref) < 1e-12
    for e in (-900, 800):   # windows that cannot be scaled take chains
        assert relerr(np.ldexp(host(G.apply_K(dev(x) * 2.0 ** e)), -e), ref) < 1e-12
    G.close()
