"""GPU: the sliced FP64 products hold every component to the bound of a chain of
DFMA, K 2^-53 Σ|a||b|, also where the elements of a row or column span far more than the
64 bits of its digits and only small ones meet: a diagonal matrix and a graded vector,
columns A e_j, wide magnitudes on both sides.  Through the matvec that takes raw
generators (U = 0), on each kernel: up to 8 columns, up to 16 on few and on many
nodes, more."""
import numpy as np
import pytest

from paper_2311_00921_gb300 import hss

pytestmark = pytest.mark.gpu
LD = np.longdouble

SHAPES = [(9, 1, 1), (60, 8, 1), (128, 1, 1), (129, 12, 1), (129, 16, 7), (257, 5, 2), (300, 33, 1),
          (70, 17, 3)]   # leaf, columns, levels


def _product(D, x, levels):
    """D x, leaf block by leaf block"""
    import torch
    nodes, leaf, nrhs = x.shape
    pack = lambda v: torch.as_tensor(np.ascontiguousarray(v.transpose(0, 2, 1))).cuda().reshape(-1)
    zero = lambda n: torch.zeros(n, dtype=torch.float64, device="cuda")
    xd = hss.colmajor(x.reshape(nodes * leaf, nrhs))
    yd = torch.zeros_like(xd.t()).t()
    hss.matvec_noalloc((nodes * leaf, leaf, 1, levels), pack(D), zero(nodes * leaf),
                       zero(max(1, 2 * (nodes - 2))), zero(nodes - 1), xd, yd)
    return yd.cpu().numpy().reshape(nodes, leaf, nrhs)


def _check(D, x, levels):
    y = _product(D, x, levels)
    ref = np.matmul(D.astype(LD), x.astype(LD))
    absum = np.matmul(np.abs(D), np.abs(x))
    # K products and sums at 2^-53 each and one addition of the (zero) basis part (a group
    # of 128 indices is within 128 2^-52.5 in the worst case, 2^-52 in the mean)
    tol = (D.shape[2] + 2) * 2.0 ** -53 * absum
    err = np.abs(y - ref)
    assert np.all(err <= tol), float((err / np.maximum(tol, 1e-300)).max())


def _rng(leaf, nrhs, seed):
    return np.random.default_rng(1000 * leaf + 10 * nrhs + seed)


@pytest.mark.parametrize("leaf,nrhs,levels", SHAPES)
def test_diagonal_matrix_and_graded_vector(leaf, nrhs, levels):
    rng = _rng(leaf, nrhs, 0)
    nodes = 1 << levels
    D = np.zeros((nodes, leaf, leaf))
    D[:, np.arange(leaf), np.arange(leaf)] = rng.standard_normal((nodes, leaf))
    grade = 2.0 ** -np.linspace(0.0, 70.0, leaf)
    x = rng.standard_normal((nodes, leaf, nrhs)) * rng.permutation(grade)[None, :, None]
    _check(D, x, levels)


@pytest.mark.parametrize("leaf,nrhs,levels", SHAPES)
def test_columns_of_a_decaying_kernel(leaf, nrhs, levels):
    """A e_j: each result is one entry, down to 2^-140 of its row's largest."""
    rng = _rng(leaf, nrhs, 1)
    nodes = 1 << levels
    d = np.abs(np.arange(leaf)[:, None] - np.arange(leaf)[None]) / leaf
    D = 2.0 ** (-140.0 * d) * (1.0 + rng.random((nodes, leaf, leaf)))
    x = np.zeros((nodes, leaf, nrhs))
    for z in range(nodes):
        x[z, rng.integers(0, leaf, nrhs), np.arange(nrhs)] = 1.0 + rng.random(nrhs)
    _check(D, x, levels)


@pytest.mark.parametrize("leaf,nrhs,levels", SHAPES)
def test_wide_magnitudes_on_both_sides(leaf, nrhs, levels):
    rng = _rng(leaf, nrhs, 2)
    nodes = 1 << levels
    wide = lambda *s: rng.standard_normal(s) * 2.0 ** rng.integers(-40, 41, s)
    D, x = wide(nodes, leaf, leaf), wide(nodes, leaf, nrhs)
    D[:, leaf // 2] = 0.0                                # a row and a column of zeros
    x[:, :, nrhs // 2] *= 0.0
    D[rng.random(D.shape) < 0.7] = 0.0                  # disjoint supports
    _check(D, x, levels)


def test_denormal_rows():
    """A row whose largest element's high word is zero."""
    rng = np.random.default_rng(3)
    D, x = rng.standard_normal((2, 40, 40)), 2.0 ** 60 * rng.random((2, 40, 3))
    D[0, 7] = np.ldexp(np.floor(rng.random(40) * 2 ** 31), -1074)
    D[1, 9, :39], D[1, 9, 39] = 0.0, np.ldexp(3.0, -1074)
    _check(D, x, 1)


@pytest.mark.parametrize("leaf,nrhs,levels", [(128, 8, 3), (256, 16, 2), (256, 24, 2), (512, 8, 1)])
@pytest.mark.parametrize("peak", [1.0, 1000.0])
def test_not_less_accurate_than_a_chain(leaf, nrhs, levels, peak):
    """Root-mean-square error against that of a sequential chain in FP64 (products
    exact, one rounding a step), for uniform rows and for rows with a large diagonal.  The
    sliced product rounds once per group of 128 indices: at most half the chain's error
    from 256 indices on, which seven digits (2^-56 of the scales' product per index, as
    much as the chain itself at these sizes) would not keep."""
    rng = _rng(leaf, nrhs, 4)
    nodes = 1 << levels
    D = rng.standard_normal((nodes, leaf, leaf))
    D[:, np.arange(leaf), np.arange(leaf)] += peak
    x = rng.standard_normal((nodes, leaf, nrhs))
    Dl, xl = D.astype(LD), x.astype(LD)
    ref = np.matmul(Dl, xl)
    chain = np.zeros(x.shape)
    for k in range(leaf):
        chain = (chain + Dl[:, :, k, None] * xl[:, None, k, :]).astype(np.float64)
    rms = lambda v: float(np.sqrt(np.mean(((v - ref).astype(np.float64)) ** 2)))
    assert rms(_product(D, x, levels)) <= (0.5 if leaf >= 256 else 1.0) * rms(chain)


@pytest.mark.parametrize("levels,leaf,rank", [(1, 96, 20), (2, 160, 40), (1, 256, 64), (2, 64, 32)])
def test_factor_of_graded_rows(levels, leaf, rank):
    """Rows that the bases do not touch, scaled down to 2^-30: no transformation mixes
    them, so the Cholesky's backward error is relative to sqrt(a_ii a_jj) whatever the
    scaling."""
    from oracle import ulv as O
    from paper_2311_00921_gb300 import inputs as I
    h = I.random_hss(levels, leaf, rank, 5)
    free = leaf - rank - 9
    scale = np.ones(leaf)
    scale[:max(free, 0)] = 2.0 ** -(30 * np.random.default_rng(1).random(max(free, 0)))
    for i in range(len(h.D)):
        h.U[i][:max(free, 0)] = 0.0
        h.D[i] = scale[:, None] * h.D[i] * scale[None]
    A = O.assemble_dense(h)
    b = np.random.default_rng(2).standard_normal((h.n, 3))
    dev = hss.HSS(h)
    dev.factorize("fp64")
    x = dev.solve(hss.colmajor(b)).cpu().numpy()
    res = np.abs(b - np.matmul(A.astype(LD), x.astype(LD)))
    d = np.sqrt(np.diag(A))
    assert np.all(res <= (3 * h.n + 1) * 2.0 ** -53 * d[:, None] * (d[None] @ np.abs(x)))
