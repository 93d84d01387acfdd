"""The server admits requests by an estimate of their peak device memory: the peak measured in the
driver's memory pool stays below the estimate, on requests whose set-up needs most of what the
estimate cannot read off the request (large stars, dense blocks past the 224 nodes whose
inverse is formed in shared memory, factor pools that grow)."""
import ctypes as C

import numpy as np
import pytest

from paper_2207_07488_gb300 import networks as nw

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2207_07488_gb300 import spnet  # noqa: E402

USED_NOW, USED_HIGH = 7, 8  # cudaMemPoolAttrUsedMemCurrent, cudaMemPoolAttrUsedMemHigh


@pytest.fixture(scope="module")
def pool():
    """pool(): (bytes of the default pool in use, their high-water mark since the last call)."""
    torch.zeros(1).cuda()
    for name in ("libcudart.so.13", "libcudart.so", "/usr/local/cuda/lib64/libcudart.so"):
        try:
            rt = C.CDLL(name)
            break
        except OSError:
            rt = None
    if rt is None:
        pytest.skip("no CUDA runtime library to ask")
    handle, v = C.c_void_p(), C.c_uint64(0)
    assert rt.cudaDeviceGetDefaultMemPool(C.byref(handle), torch.cuda.current_device()) == 0

    def get(attr):
        assert rt.cudaMemPoolGetAttribute(handle, attr, C.byref(v)) == 0
        return v.value

    def read():
        torch.cuda.synchronize()
        now, high, zero = get(USED_NOW), get(USED_HIGH), C.c_uint64(0)
        assert rt.cudaMemPoolSetAttribute(handle, USED_HIGH, C.byref(zero)) == 0
        return now, high
    return read


def _net(kind):
    if kind == "2d":
        return nw.fiber_network_2d(10000, 0.1, 77)
    return nw.fiber_network_3d(40000, 0.1, 0.004, 3000, keep="clamped_x" if kind == "truss" else "dirichlet_x")


CASES = [("2d", 16, 224, 1, "mixed"), ("2d", 16, 224, 1, "fp64"), ("2d", 40, 0, 8, "mixed"), ("truss", 8, 224, 1, "mixed"),
         ("truss", 12, 0, 2, "fp64"), ("3d", 16, 0, 1, "mixed"), ("3d", 8, 0, 1, "fp64")]


@pytest.mark.parametrize("kind,nH,block,k,prec", CASES)
def test_the_peak_stays_below_the_estimate(pool, kind, nH, block, k, prec):
    net = _net(kind)
    p = nw.truss_band_problem(net, 1.0 / nH) if kind == "truss" else nw.scalar_band_problem(net, 1.0 / nH)
    pr = spnet.PREC_FP64 if prec == "fp64" else spnet.PREC_MIXED
    if block:
        op = spnet.Operator.from_problem(p)
        pc = spnet.Preconditioner(op, p.H, p.gamma_faces, precision=pr)
        assert pc.export(spnet.EXPORT_STAR_CORE).max() > block
        pc.close()
        op.close()
    F = np.random.default_rng(1).uniform(0.0, 1.0, (k, p.n_dof))
    est = spnet.request_estimate(p, f=F, precision=pr, batch_rhs=k)
    sv = spnet.Server(max_inflight=1)
    held, _ = pool()  # by handles of other tests
    _, res = sv.wait(sv.submit(p, f=F, precision=pr, batch_rhs=k))
    peak = pool()[1] - held
    sv.close()
    assert res["status"] == spnet.OK, res["message"]
    assert 0 < peak <= est
