"""Stars whose dense block passes the size limit of the inverse and fails its condition limit are
factored again, they alone: a network of two clusters, each within one element of the mesh, of
which the left has conductances over eight decades and is all but free (its blocks cannot be kept
as rounded inverses) and the right is well conditioned."""
import numpy as np
import pytest

from paper_2207_07488_gb300 import networks as nw

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2207_07488_gb300 import spnet  # noqa: E402

H = 0.25


def _clusters(n, seed):
    """n nodes in element (0, 1) and n in element (3, 1), each joined to random others of its cluster and to a
    Dirichlet node; the problem, K on the free nodes, coordinates."""
    rng = np.random.default_rng(seed)
    X = rng.uniform(0.27, 0.48, (2 * n, 2))
    X[:n, 0] = rng.uniform(0.02, 0.23, n)
    X[n:, 0] = rng.uniform(0.77, 0.98, n)
    i = np.repeat(np.arange(2 * n), 40)
    j = rng.integers(0, n, 80 * n) + n * (i >= n)
    E = np.unique(np.sort(np.stack([i, j], 1)[i != j], axis=1), axis=0)
    left = E[:, 0] < n
    c = np.where(left, 10.0 ** rng.uniform(-4.0, 4.0, len(E)), rng.uniform(0.5, 2.0, len(E)))
    E = np.concatenate([E, np.stack([np.arange(2 * n), np.full(2 * n, 2 * n)], 1)])
    c = np.concatenate([c, np.where(np.arange(2 * n) < n, 1e-6, 0.5)])
    m = len(E)
    net = nw.Network(2, np.concatenate([X, [[0.0, 0.5]]]), E.astype(np.int64), np.zeros(m, np.int8), c, c,
                     np.zeros((m, 2)), (1.0, 1.0))
    p = nw.Problem(net, 1, "scalar", np.array([2 * n], np.int64), np.zeros(1), np.ones(2 * n + 1), H, (0,))
    K = np.zeros((2 * n + 1,) * 2)
    for (a, b), w in zip(E, c):
        K[[a, b], [b, a]] -= w
        K[[a, b], [a, b]] += w
    return p, K[:-1, :-1], X


def test_marked_stars_are_done_again_alone():
    n = 300
    p, A, X = _clusters(n, 11)
    op = spnet.Operator.from_problem(p)
    spnet.profile_reset()
    spnet.profile_enable(True)
    pc = spnet.Preconditioner(op, H, p.gamma_faces)
    launches = spnet.profile_read()
    spnet.profile_enable(False)
    flat = spnet.Preconditioner(op, H, p.gamma_faces, panels=False)  # no star's block inverted
    lev = [q.export(spnet.EXPORT_STAR_LEVELS) for q in (pc, flat)]
    assert pc.info.n_stars == 4 and pc.export(spnet.EXPORT_STAR_CORE).min() >= 32
    # the levels of a factorisation without inverses in the left stars only
    assert (lev[0] <= lev[1]).all() and sorted(lev[0] == lev[1]) == [False] * 2 + [True] * 2
    # one pass over all stars, one over the marked ones with the scratch they need
    assert launches["star_symbolic"][0] == 2 and launches["star_numeric"][0] == 2
    r = np.random.default_rng(1).standard_normal(2 * n)
    rl, rr = np.where(np.arange(2 * n) < n, r, 0.0), np.where(np.arange(2 * n) < n, 0.0, r)
    # the marked stars are those of a set-up without inverses
    np.testing.assert_array_equal(pc.stars(rl), flat.stars(rl))
    # the others keep their factors and inverses
    el = np.floor(X / H).astype(int)
    want = np.zeros(2 * n)
    for y in np.ndindex(3, 3):
        on = np.nonzero(((el == y) | (el == np.add(y, 1))).all(axis=1) & (np.arange(2 * n) >= n))[0]
        if on.size:
            want[on] += np.linalg.solve(A[np.ix_(on, on)], rr[on])
    assert np.linalg.norm(pc.stars(rr) - want) <= 2e-4 * np.linalg.norm(want)
    flat.close()
    pc.close()
    op.close()


def _nearly_singular(n, seed):
    """A complete graph of n nodes in one star, tied to its Dirichlet node by less than the
    rounding of its diagonal: whether the last pivot comes out positive is the rounding's choice."""
    rng = np.random.default_rng(seed)
    i, j = np.triu_indices(n, 1)
    E = np.concatenate([np.stack([i, j], 1), [[0, n]]])
    c = np.concatenate([rng.uniform(0.5, 2.0, len(i)), [1e-15]])
    X = np.concatenate([rng.uniform(0.1, 0.9, (n, 2)), [[0.0, 0.5]]])
    net = nw.Network(2, X, E.astype(np.int64), np.zeros(len(E), np.int8), c, c, np.zeros((len(E), 2)), (1.0, 1.0))
    return nw.Problem(net, 1, "scalar", np.array([n], np.int64), np.zeros(1), np.ones(n + 1), 0.5, (0,))


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_a_pivot_lost_in_the_inverse_does_not_refuse_a_star_that_factors(prec):
    pr = spnet.PREC_FP64 if prec == "fp64" else spnet.PREC_MIXED
    taken = {True: 0, False: 0}
    for seed in range(40):
        p = _nearly_singular(40, seed)
        op = spnet.Operator.from_problem(p)
        ok = {}
        for panels in (True, False):
            try:
                spnet.Preconditioner(op, 0.5, p.gamma_faces, precision=pr, panels=panels).close()
                ok[panels] = True
            except spnet.SpnetError as e:
                assert e.code == spnet.ERR_NOT_SPD
                ok[panels] = False
        assert ok[True] or not ok[False], seed
        taken[ok[False]] += 1
        op.close()
    assert taken[True] > 0 and taken[False] > 0  # both outcomes of the factorisation were met
