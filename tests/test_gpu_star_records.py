"""The star solves (Section 4.1, eq. defPj) at the edges of their record format: one star that
holds every free dof (H = 1/2 on the unit square), its local problem solved in numpy.

The graphs put the dense block that ends the elimination at the sizes where its rows and
columns fall into other row blocks, records and record sizes (1..33 nodes, 100, 225 on the
other side of the shared-memory inverse, 300 and 600 for larger records), make rows longer
than one group takes (a hub; without inverses, the rows of the block), and stars that are one
dof or all dense block.  Several right-hand sides: every count that changes the vector width or
leaves it ragged.

Bounds: FP64 every entry within 1e-9 of the largest (the local condition numbers stay below
1e5: rounding 1e-11); FP32 factors 2e-4 of the norm (the mixed bound of the parity tests)."""
import numpy as np
import pytest

from paper_2207_07488_gb300 import networks as nw

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2207_07488_gb300 import spnet  # noqa: E402


def _edges(kind, n, rng):
    if kind == "sparse":  # a tree and a few more edges: many rounds, a small dense block
        a = np.arange(1, n)
        e = np.stack([a, (a * rng.random(n - 1)).astype(int)], 1)
        x = rng.integers(0, n, (n // 4, 2))
        return np.concatenate([e, x[x[:, 0] != x[:, 1]]])
    if kind == "hub":  # one node joined to 120 others, chains between them
        a = np.arange(1, n)
        e = np.stack([a, a - 1], 1)
        return np.concatenate([e, np.stack([np.full(min(120, n - 1), n // 2), rng.permutation(n)[:min(120, n - 1)]], 1)])
    # "dense": every pair, or (a row of K holds at most 128 entries) 50 neighbours on either side
    i, j = np.triu_indices(n, 1)
    near = np.minimum(j - i, n - (j - i)) <= 50
    return np.stack([i, j], 1)[near]


def _star(kind, n, seed):
    """A scalar problem whose one star holds n free dofs, and its local matrix."""
    rng = np.random.default_rng(seed)
    E = _edges(kind, n, rng)
    E = E[E[:, 0] != E[:, 1]]
    E = np.unique(np.sort(E, axis=1), axis=0)
    E = np.concatenate([E, np.stack([np.arange(n), np.full(n, n)], 1)])  # each tied to a Dirichlet node
    c = rng.uniform(0.5, 2.0, len(E))
    c[-n:] = 0.1
    X = np.concatenate([rng.uniform(0.1, 0.9, (n, 2)), [[0.0, 0.5]]])
    m = len(E)
    net = nw.Network(2, X, E.astype(np.int64), np.zeros(m, np.int8), c, c, np.zeros((m, 2)), (1.0, 1.0))
    p = nw.Problem(net, 1, "scalar", np.array([n], np.int64), np.zeros(1), np.ones(n + 1), 0.5, (0,))
    K = np.zeros((n + 1, n + 1))
    for (i, j), w in zip(E, c):
        K[i, j] -= w
        K[j, i] -= w
        K[i, i] += w
        K[j, j] += w
    return p, K[:n, :n]


CASES = [("sparse", n) for n in (1, 2, 31, 32, 33, 40, 300, 900)] + [("hub", 400), ("hub", 1500)] + \
        [("dense", n) for n in (4, 5, 33, 100, 129, 225, 300, 600)]


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("kind,n", CASES)
def test_star_solve(kind, n, prec):
    p, A = _star(kind, n, 100 + n)
    op = spnet.Operator.from_problem(p)
    pr = spnet.PREC_FP64 if prec == "fp64" else spnet.PREC_MIXED
    ref = {}
    for panels in (True, False):  # the inverse of the dense block; the block a node a level
        pc = spnet.Preconditioner(op, 0.5, p.gamma_faces, precision=pr, batch_rhs=4, panels=panels)
        assert pc.info.n_stars == 1 and pc.info.max_star == n
        R = np.random.default_rng(n).standard_normal((33, n))
        want = np.linalg.solve(A, R.T).T
        for k in (1, 2, 3, 5, 32):
            Z = pc.apply_batch(R[:k], which=2)
            for j in range(k):
                d = np.abs(Z[j] - want[j])
                if prec == "fp64":
                    assert d.max() <= 1e-9 * np.abs(want[j]).max(), (k, j)
                else:
                    assert np.linalg.norm(d) <= 2e-4 * np.linalg.norm(want[j]), (k, j)
            ref.setdefault(panels, {})[k] = Z
        z = pc.stars(R[0])
        # the same records and the same order of sums whatever the right-hand sides beside it
        for k in (1, 2, 3, 5, 32):
            np.testing.assert_array_equal(z, ref[panels][k][0])
        for w in (1, 2, 8):  # and whatever the warps that share the star
            pw = spnet.Preconditioner(op, 0.5, p.gamma_faces, precision=pr, star_map=w, panels=panels)
            np.testing.assert_array_equal(z, pw.stars(R[0]))
            pw.close()
        pc.close()
    op.close()


def test_dense_block_beyond_the_inverse():
    # a band of 100 neighbours around a ring of 1400 nodes leaves a block past the 1024 nodes
    # that are inverted: it is eliminated a node a level (long rows across the lanes)
    n = 1400
    p, A = _star("dense", n, 7)
    op = spnet.Operator.from_problem(p)
    pc = spnet.Preconditioner(op, 0.5, p.gamma_faces, precision=spnet.PREC_FP64)
    assert pc.export(spnet.EXPORT_STAR_CORE)[0] > 1024
    r = np.random.default_rng(3).standard_normal(n)
    want = np.linalg.solve(A, r)
    assert np.abs(pc.stars(r) - want).max() <= 1e-9 * np.abs(want).max()
