"""SPNET_ERR_TIMEOUT: the star solves wait for their factor data with a limit, which the tests
set to nothing, so that every such wait of a healthy solve gives up and the call returns the
status; with the limit put back the same handles work again, with the results they gave before."""
import numpy as np
import pytest

from paper_2207_07488_gb300 import networks as nw

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2207_07488_gb300 import spnet  # noqa: E402


def _timeout(call):
    with pytest.raises(spnet.SpnetError) as e:
        call()
    assert e.value.code == spnet.ERR_TIMEOUT


@pytest.fixture
def handles():
    p = nw.scalar_band_problem(nw.fiber_network_2d(400, 0.1, seed=7), 0.25)
    op = spnet.Operator.from_problem(p)
    pc = spnet.Preconditioner(op, p.H, p.gamma_faces, batch_rhs=3)
    yield p, op, pc
    op.wait_limit()
    pc.close()
    op.close()


def test_every_call_with_star_solves_reports_a_wait_that_ran_out(handles):
    p, op, pc = handles
    F, G = np.tile(p.f, (3, 1)) + 1.0, np.tile(p.dirichlet_vals, (3, 1))
    calls = [lambda: spnet.pcg_solve(op, pc, p.f, p.dirichlet_vals)[0], lambda: spnet.pcg_solve(op, pc, F, G)[0]]
    before = [c() for c in calls]
    r = np.random.default_rng(1).standard_normal((3, op.info.n_free))
    op.wait_limit(0)
    for c in calls + [lambda: pc.apply(r[0]), lambda: pc.stars(r[0]), lambda: pc.apply_batch(r)]:
        _timeout(c)
    assert np.isfinite(pc.apply_batch(r, which=1)).all()  # no star solve in it
    op.wait_limit()
    for c, b in zip(calls, before):
        np.testing.assert_array_equal(c(), b)


@pytest.mark.parametrize("failing", ["solve", "apply", "stars"])
def test_an_apply_after_a_timeout_reports_its_own_waits_only(handles, failing):
    p, op, pc = handles
    r = np.random.default_rng(2).standard_normal(op.info.n_free)
    z, w = pc.apply(r), pc.stars(r)
    op.wait_limit(0)
    _timeout({"solve": lambda: spnet.pcg_solve(op, pc, p.f, p.dirichlet_vals),
              "apply": lambda: pc.apply(r), "stars": lambda: pc.stars(r)}[failing])
    op.wait_limit()
    np.testing.assert_array_equal(pc.apply(r), z)
    np.testing.assert_array_equal(pc.stars(r), w)


@pytest.mark.parametrize("opts", [dict(), dict(star_map=4, batch_rhs=4)], ids=["warps", "columns"])
def test_a_setup_whose_timed_solves_ran_out_fails_and_keeps_no_choice(opts):
    # enough stars (four an SM) for the choice of warps to be timed
    p = nw.scalar_band_problem(nw.fiber_network_2d(1000, 0.1, seed=7), 1.0 / 40)
    op = spnet.Operator.from_problem(p)
    spnet.tune_cache_clear()
    op.wait_limit(0)
    _timeout(lambda: spnet.Preconditioner(op, p.H, p.gamma_faces, **opts))
    assert spnet.tune_counts() == (0, 0)
    op.wait_limit()
    pc = spnet.Preconditioner(op, p.H, p.gamma_faces, **opts)
    assert pc.info.n_stars >= 4 * torch.cuda.get_device_properties(0).multi_processor_count
    assert spnet.tune_counts() == (1, 0)
    assert np.isfinite(pc.apply(np.ones(op.info.n_free))).all()
    pc.close()
    op.close()


def test_a_negative_limit_is_refused(handles):
    _, op, _ = handles
    with pytest.raises(spnet.SpnetError) as e:
        op.wait_limit(-1)
    assert e.value.code == spnet.ERR_BAD_INPUT
