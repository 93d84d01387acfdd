"""A tuner cache saved by an earlier build holds choices of kernels that are gone, as kinds 0 and 2:
they load and are not taken for the present kernels' choices, which are measured."""
import pytest

from paper_2207_07488_gb300 import networks as nw

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2207_07488_gb300 import spnet  # noqa: E402


def test_choices_of_earlier_kernels_are_not_taken(tmp_path):
    # enough stars for the choice of warps to be timed
    p = nw.scalar_band_problem(nw.fiber_network_2d(1000, 0.1, seed=7), 1.0 / 40)
    op = spnet.Operator.from_problem(p)
    path = tmp_path / "tune.tsv"

    def choices():
        spnet.Preconditioner(op, p.H, p.gamma_faces, batch_rhs=4).close()
        spnet.tune_cache_save(str(path))
        return [line.split("\t") for line in path.read_text().splitlines()]

    spnet.tune_cache_clear()
    now = choices()
    assert sorted(int(kind) for _, kind, _, _ in now) == [3, 4] and spnet.tune_counts() == (2, 0)
    old = [[dev, {"3": "0", "4": "2"}[kind], cls, "1"] for dev, kind, cls, _ in now]
    path.write_text("".join("\t".join(line) + "\n" for line in old))
    spnet.tune_cache_clear()
    spnet.tune_cache_load(str(path))
    assert sorted(int(kind) for _, kind, _, _ in choices()) == [0, 2, 3, 4]
    assert spnet.tune_counts() == (2, 0)
    spnet.tune_cache_clear()
    op.close()
