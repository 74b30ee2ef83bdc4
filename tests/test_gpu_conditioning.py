"""GPU: FP64 solves of badly conditioned matrices (smooth 1-D covariances with a small
nugget, condition numbers 1e6 to 4e12) leave residuals like those of triangular
substitution: the products with inverted diagonal blocks are corrected."""
import numpy as np
import pytest
import scipy.linalg as sla

from oracle import ulv as O
from paper_2311_00921_gb300 import hss
from paper_2311_00921_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def gaussian_line(levels, leaf, rank, nugget):
    """exp(-(d / 0.3)²) + nugget on sorted points of the unit interval, whose far blocks have
    numerical rank far below `rank`."""
    n, nl = leaf << levels, 1 << levels
    x = np.sort(np.random.default_rng(0).random(n))
    A = np.exp(-((x[:, None] - x[None]) / 0.3) ** 2) + nugget * np.eye(n)
    rows = lambda l, i: np.arange(i * (n >> l), (i + 1) * (n >> l))
    far = lambda l, i: np.delete(A[rows(l, i)], rows(l, i), axis=1)
    basis = {levels: [np.linalg.svd(far(levels, i))[0][:, :rank] for i in range(nl)]}
    E = {}
    for l in range(levels - 1, 0, -1):
        E[l], basis[l] = [], []
        for i in range(1 << l):
            W = sla.block_diag(*basis[l + 1][2 * i:2 * i + 2])
            E[l].append(np.linalg.svd(W.T @ far(l, i))[0][:, :rank])
            basis[l].append(W @ E[l][-1])
    S = {l: [basis[l][2 * k + 1].T @ A[np.ix_(rows(l, 2 * k + 1), rows(l, 2 * k))] @ basis[l][2 * k]
             for k in range(1 << (l - 1))] for l in range(1, levels + 1)}
    D = [A[np.ix_(rows(levels, i), rows(levels, i))] for i in range(nl)]
    return I.HSSMatrix(levels=levels, sizes=np.full(nl, leaf), D=D, U=basis[levels], E=E, S=S,
                       ranks={l: np.full(1 << l, rank) for l in range(1, levels + 1)})


@pytest.mark.parametrize("nugget", [1e-4, 1e-6, 1e-8, 1e-10])
@pytest.mark.parametrize("levels,leaf,rank", [(1, 256, 32), (2, 300, 20), (3, 96, 33), (1, 200, 12),
                                              (1, 128, 80)])
def test_residual_like_substitution(levels, leaf, rank, nugget):
    h = gaussian_line(levels, leaf, rank, nugget)
    A = O.assemble_dense(h).astype(np.longdouble)
    b = I.rhs(h.n, 8, 1)
    norm = lambda x: float((np.linalg.norm((A @ x - b).astype(float), axis=0)
                            / np.linalg.norm(b, axis=0)).max())
    plain = norm(O.solve(O.factor(h), b))
    dev = hss.HSS(h)
    dev.factorize("fp64")
    bd = hss.colmajor(b)
    batch = hss.HSSBatch([h, h])
    batch.factorize()
    # two realisations of the same rounding errors: each within a small factor of the other
    assert norm(dev.solve(bd).cpu().numpy()) <= 4.0 * plain
    assert norm(batch.solve([bd, bd])[1].cpu().numpy()) <= 4.0 * plain


def test_one_badly_conditioned_leaf_among_others():
    """Nodes of a level that need corrections beside nodes that do not: without coupling
    each leaf is solved as in a matrix whose leaves are all of its kind (the sibling of
    the badly conditioned one excepted: the parent's basis mixes the two)."""
    def residuals(shifts):
        h = gaussian_line(2, 200, 24, 1e-8)
        h.D = [d + s * np.eye(200) for d, s in zip(h.D, shifts)]
        h.S = {l: [0.0 * s for s in h.S[l]] for l in h.S}
        b = I.rhs(h.n, 5, 1)
        dev = hss.HSS(h)
        dev.factorize("fp64")
        batch = hss.HSSBatch([h])
        batch.factorize()
        bd = hss.colmajor(b)
        out = []
        for x in (dev.solve(bd), batch.solve([bd])[0]):
            x = x.cpu().numpy().reshape(4, 200, 5)
            out.append([np.linalg.norm((h.D[i].astype(np.longdouble) @ x[i]
                                        - b[200 * i:200 * (i + 1)]).astype(float)) for i in range(4)])
        return np.array(out)

    mixed, bad, good = residuals([0, 2, 2, 2]), residuals([0] * 4), residuals([2] * 4)
    assert np.all(mixed[:, 0] <= 4.0 * bad[:, 0])
    assert np.all(mixed[:, 2:] <= 4.0 * good[:, 2:])
