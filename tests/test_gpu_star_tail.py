"""Where the elimination of a star stops for its dense block: at an eighth of its dofs, at most 128, or
64 on 3D networks of few stars (the inverse of a larger block is waited for).  The star term on both
sides of the rule against the oracle (Section 4.1, eq. defPj), with the bounds of the parity tests."""
import numpy as np
import pytest

from oracle.solve import OracleSolver
from paper_2207_07488_gb300 import networks as nw

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from parity_checks import check_star_term  # noqa: E402

from paper_2207_07488_gb300 import spnet  # noqa: E402

CASES = {"3d, 1 star": (3, 8000, 2, 64), "3d, 8 stars": (3, 16000, 3, 64), "3d, 64 stars": (3, 24000, 5, 128),
         "2d, 9 stars": (2, 1000, 4, 128)}


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("name", list(CASES))
def test_the_size_of_the_dense_block(name, prec):
    dim, size, nH, most = CASES[name]
    net = nw.fiber_network_2d(size, 0.1, 1000 + size) if dim == 2 else nw.fiber_network_3d(size, 0.1, 0.004, 2000 + size)
    p = nw.scalar_band_problem(net, 1.0 / nH)
    op = spnet.Operator.from_problem(p)
    pc = spnet.Preconditioner(op, p.H, p.gamma_faces,
                              precision=spnet.PREC_FP64 if prec == "fp64" else spnet.PREC_MIXED)
    n, core = pc.export(spnet.EXPORT_STAR_SIZES), pc.export(spnet.EXPORT_STAR_CORE)
    assert n.max() >= 8 * most
    # (smaller where a round of the elimination goes past the mark)
    assert core.max() <= most and (most == 64 or np.median(core[n >= 8 * most]) > 64)
    o = OracleSolver(p)
    r = np.random.default_rng(3).standard_normal(op.info.n_free)
    check_star_term(o, r, pc.stars(r), prec)
    pc.close()
    op.close()
