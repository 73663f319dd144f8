"""State norms (tqc_hss_norms) at the edges of the kernel's splits: no
outputs, no cuts, fewer than 32 states, and rows split over every cluster
size, against NumPy in FP64.

Bound: a norm is the root of a sum of n squares, each rounded once and added
in some order: relative error at most (n + 3) 2^-53."""
import numpy as np
import pytest

from gen import Network, Node

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2502_03445_gb300 import tqc  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("cuts,outs", [(0, 3), (0, 9), (1, 0), (1, 12), (2, 5), (3, 1), (3, 6), (4, 7), (5, 2), (5, 11),
                                       (6, 0), (6, 4), (6, 7), (6, 10), (7, 5)])
def test_norms(cuts, outs, dtype):
    rng = np.random.Generator(np.random.PCG64(100 * cuts + outs))
    mine = list(range(cuts))
    a = rng.standard_normal((4 ** cuts, 1 << outs)).astype(dtype)
    nodes = [Node(list(range(outs)), mine, [0] * cuts, a.reshape(-1)),
             Node([outs], mine, [1] * cuts, rng.standard_normal((4 ** cuts) * 2).astype(dtype))]
    h = tqc.Network(Network(outs + 1, cuts, nodes), dtype=tqc.F64 if dtype == np.float64 else tqc.F32)
    out = torch.full((1 << outs,), float("nan"), dtype=torch.float64, device="cuda")
    h.hss_norms(0, out)
    want = np.sqrt((a.astype(np.longdouble) ** 2).sum(0)).astype(np.float64)
    np.testing.assert_allclose(out.cpu().numpy(), want, rtol=(4 ** cuts + 3) * 2.0 ** -53, atol=0)
    h.close()


# few states and many rows: the rows go over several clusters, whose sums a
# second kernel adds (fewer and more parts than lanes, and a tensor beyond L2)
@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("cuts,outs", [(8, 2), (8, 3), (9, 0), (9, 4), (9, 6), (11, 1), (8, 9)])
def test_norms_in_parts(cuts, outs, dtype):
    test_norms(cuts, outs, dtype)
