"""GPU: the FP64 products on the tensor cores (exact slicing), through the matvec
that takes raw generators, against extended precision at the edges of the tiles
(64 rows, 8 / 16 / 32 columns, 32 and 128 inner indices), and with values that the
slicing leaves to the FP64 pipe."""
import numpy as np
import pytest

from paper_2311_00921_gb300 import hss

pytestmark = pytest.mark.gpu
LD = np.longdouble


def _gen(leaf, rank, seed, spread):
    rng = np.random.default_rng(seed)
    f = lambda *s: rng.standard_normal(s) * 2.0 ** rng.integers(-spread, spread + 1, s)
    return f(2, leaf, leaf), f(2, leaf, rank), f(1, rank, rank)


def _chain(D, U, S, x, T, a=lambda v: v):
    """y = A x (levels = 1) in arithmetic T, of a(entries)."""
    D, U, S, x = (a(v).astype(T) for v in (D, U, S, x))
    h = U.transpose(0, 2, 1) @ x
    y = np.stack([S[0].T @ h[1], S[0] @ h[0]])
    return D @ x + U @ y


def _run(D, U, S, x):
    import torch
    leaf, rank, nrhs = D.shape[1], U.shape[2], x.shape[2]
    pack = lambda v: torch.as_tensor(np.ascontiguousarray(v.transpose(0, 2, 1))).cuda().reshape(-1)
    xd = hss.colmajor(x.reshape(2 * leaf, nrhs))
    yd = torch.zeros_like(xd.t()).t()
    e = torch.zeros(1, dtype=torch.float64, device="cuda")
    hss.matvec_noalloc((2 * leaf, leaf, rank, 1), pack(D), pack(U), e, pack(S), xd, yd)
    return yd.cpu().numpy().reshape(2, leaf, nrhs)


@pytest.mark.parametrize("leaf,rank,nrhs,spread", [
    (1, 1, 1, 0), (9, 9, 17, 3), (31, 16, 8, 0), (33, 32, 9, 20), (64, 24, 33, 0), (65, 10, 16, 8),
    (129, 128, 5, 0), (200, 64, 40, 12), (300, 33, 2, 0)])
def test_products_against_extended_precision(leaf, rank, nrhs, spread):
    D, U, S = _gen(leaf, rank, 10 * leaf + nrhs, spread)
    x = np.random.default_rng(leaf).standard_normal((2, leaf, nrhs))
    y = _run(D, U, S, x)
    ref = _chain(D, U, S, x, LD)
    # every product: one rounding per group of 128 inner indices and one or two at
    # the end, 2^-53 of the partial sums each; cut operands and dropped digit
    # products, 2^-58 of the largest magnitudes each; four products in a chain
    groups = sum((k + 127) // 128 + 2 for k in (leaf, rank, rank, leaf))
    absum = _chain(D, U, S, x, np.float64, np.abs)
    top = np.abs(D).max() * np.abs(x).max() * leaf
    top += (np.abs(U).max() ** 2 * np.abs(S).max() * np.abs(x).max()) * leaf * rank * rank
    tol = groups * 2.0 ** -53 * absum + 4 * 2.0 ** -58 * top
    assert np.all(np.abs(y - ref) <= tol), float((np.abs(y - ref) / tol).max())


def test_values_outside_the_sliced_range():
    """Infinities, NaN, overflow and tiny magnitudes as in the plain product; other
    columns unharmed."""
    leaf, rank, nrhs = 70, 20, 12
    D, U, S = _gen(leaf, rank, 5, 0)
    x = np.random.default_rng(6).standard_normal((2, leaf, nrhs))
    D, x = np.abs(D), np.abs(x)
    U[:] = 0.0
    x[0, 3, 1], x[1, 69, 2], x[0, 0, 4] = np.inf, np.nan, -np.inf
    D[1, 5, 7], x[1, 7, 6] = 1e200, 1e200          # overflows in row 5, column 6
    x[:, :, 9] *= 1e-290                            # below the sliced range
    x[:, :, 10] = 0.0
    y = _run(D, U, S, x)
    with np.errstate(all="ignore"):
        plain = _chain(D, U, S, x, np.float64)   # also 0 * inf and 0 * NaN in U's products
    special = np.where(np.isfinite(plain), 0.0, plain)
    np.testing.assert_array_equal(np.where(np.isfinite(y), 0.0, y), special)
    assert np.all(y[0, :, 1] == np.inf) and np.all(np.isnan(y[:, :, 2])) and y[1, 5, 6] == np.inf
    assert np.all(y[:, :, 10] == 0.0)
    for j in (0, 3, 5, 7, 8, 9, 11):
        ref = np.einsum("zij,zj->zi", D.astype(LD), x[:, :, j].astype(LD))
        assert np.all(np.abs(y[:, :, j] - ref) <= (leaf + 4) * 2.0 ** -53 * np.abs(ref)), j


@pytest.mark.parametrize("leaf,rank,nrhs", [
    (18, 17, 1), (49, 17, 3), (81, 17, 16), (82, 17, 17), (145, 17, 2), (146, 18, 9),
    (300, 40, 5), (256, 130, 1), (20, 20, 4)])
def test_blocked_levels_against_oracle(leaf, rank, nrhs):
    """The FP64 level routines at the edges of their blocks (1, 32, 64, 128 and more
    eliminated columns, ragged ones, none), with the tolerances of the parity tests."""
    from oracle import ulv as O
    from paper_2311_00921_gb300 import inputs as I
    h = I.random_hss(3, leaf, rank, seed=leaf + rank, orthonormal=False)
    F, b = O.factor(h), I.rhs(h.n, nrhs, 7)
    x_ref, ld_ref = O.solve(F, b), O.logdet(F)
    dev = hss.HSS(h)
    dev.factorize("fp64")
    x = dev.solve(hss.colmajor(b)).cpu().numpy()
    err = np.linalg.norm(x - x_ref, axis=0) / np.linalg.norm(x_ref, axis=0)
    assert err.max() <= 1e-10
    assert abs(dev.logdet() - ld_ref) <= 1e-12 * abs(ld_ref)


def test_pivot_in_a_later_block():
    """A block whose first non-positive pivot lies past the first 64 columns is
    reported at the oracle's column."""
    from oracle import ulv as O
    from paper_2311_00921_gb300 import inputs as I
    h = I.random_hss(2, 200, 20, seed=9)
    h.D[2][150, 150] *= -1.0
    dev = hss.HSS(h)
    dev.factorize("fp64")
    assert dev.last_info()["code"] == -3
    with pytest.raises(O.NotSPD) as eo:
        O.factor(h)
    info = dev.last_info()
    assert (info["level"], info["node"], info["col"]) == (eo.value.level, eo.value.node,
                                                         eo.value.col)
    assert info["col"] > 64


@pytest.mark.parametrize("leaf,rank,nrhs", [
    (1, 1, 8), (15, 15, 9), (16, 7, 16), (17, 17, 1), (127, 33, 8), (128, 4, 7), (257, 40, 3),
    (1300, 5, 8), (1300, 5, 16), (2500, 2, 8)])
def test_narrow_products_against_extended_precision(leaf, rank, nrhs):
    """Right-hand sides of up to 8 and 16 columns at the edges of the narrow kernel's
    tiles (16 rows, 32 indices a warp, one and two groups at a time)."""
    test_products_against_extended_precision(leaf, rank, nrhs, 6)


def test_batch_levels_against_oracle():
    """A forest whose heights hold both kinds of parents, at ranks below, at and above
    the blocks of the level routines, with nothing eliminated at some leaves."""
    from oracle import ulv as O
    from paper_2311_00921_gb300 import inputs as I
    mats = [I.random_hss(L, leaf, r, seed=50 + i, orthonormal=False) for i, (L, leaf, r) in
            enumerate([(3, 90, 17), (1, 90, 17), (2, 90, 17), (2, 24, 24), (1, 24, 24),
                       (2, 200, 130), (1, 200, 130), (2, 300, 9)])]
    bs = [I.rhs(h.n, 3, 60 + i) for i, h in enumerate(mats)]
    bt = hss.HSSBatch(mats)
    bt.factorize()
    xs, lds = bt.solve([hss.colmajor(b) for b in bs]), bt.logdet()
    for h, b, x, ld in zip(mats, bs, xs, lds):
        F = O.factor(h)
        x_ref, ld_ref = O.solve(F, b), O.logdet(F)
        err = np.linalg.norm(x.cpu().numpy() - x_ref, axis=0) / np.linalg.norm(x_ref, axis=0)
        assert err.max() <= 1e-10
        assert abs(ld - ld_ref) <= 1e-12 * abs(ld_ref)
