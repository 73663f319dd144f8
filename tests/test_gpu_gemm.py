"""CUDA-core FP32 steps with K >= 16 (whole 128 x 128, 128 x 64 and 64 x 64
tiles, 16 k at a time; 32 x 32 tiles or parts of them, 64 k at a time) against the FP64 oracle, element by element.

Bound: a result is one chain of K fused multiply-adds (K roundings), its
operands are FP64 inputs rounded once each, and the scale and the scaled
result round twice more: |error| <= (K + 8) 2^-24 sum_k |a_k| |b_k|, the sum
being the oracle's own value on the tensors' absolute values."""
import numpy as np
import pytest

import oracle
from gen import Network, Node, tensors

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2502_03445_gb300 import tqc  # noqa: E402

SIMT_64x64, SIMT_128x128, SIMT_128x64, SIMT_32x32 = 0, 1, 2, 4


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


# (rows, columns, cuts, where the row qubits sit, tile): one chunk of K (16)
# and several; one tile, fewer and more tiles than the grid
CASES = [(6, 6, 3, "low", SIMT_32x32), (7, 6, 3, "mixed", SIMT_32x32), (9, 7, 4, "high", SIMT_32x32),
         (1, 0, 3, "low", SIMT_32x32), (4, 3, 4, "mixed", SIMT_32x32), (2, 7, 5, "high", SIMT_32x32),
         (14, 1, 2, "mixed", SIMT_32x32), (16, 5, 3, "mixed", SIMT_32x32),
         (15, 6, 3, "mixed", SIMT_64x64), (14, 6, 2, "high", SIMT_64x64),
         (16, 6, 3, "mixed", SIMT_128x64), (17, 6, 2, "high", SIMT_128x64), (11, 11, 2, "low", SIMT_128x128),
         (13, 10, 3, "mixed", SIMT_128x128), (15, 7, 4, "high", SIMT_128x128), (5, 9, 3, "mixed", None)]


@pytest.mark.parametrize("rows,cols,cuts,where,tile", CASES)
@pytest.mark.parametrize("out_dtype", [torch.float32, torch.float64])
def test_gemm_tiles(rows, cols, cuts, where, tile, out_dtype):
    n = rows + cols
    if where == "mixed":
        first = sorted(int(q) for q in np.random.Generator(np.random.PCG64(n)).permutation(n)[:rows])
    else:
        first = list(range(rows)) if where == "low" else list(range(cols, n))
    rest = [q for q in range(n) if q not in first]
    net = tensors.pseudo_physical_network(n, [(0, 1)] * cuts, [first, rest], 5000 + n + cuts)
    absnet = Network(n, cuts, [Node(nd.out_qubits, nd.cut_ids, nd.cut_role, np.abs(nd.data)) for nd in net.nodes])
    z = oracle.total_mass(net)
    want, terms = oracle.recon_bin_pairwise(net) / z, oracle.recon_bin_pairwise(absnet) / abs(z)
    h = tqc.Network(net)
    # the general tiles also where K = 16 would take the small-K tile
    p = tqc.Plan(h, precision="fp32", flags=tqc.FLAG_NO_SMALLK)
    out = torch.full((p.out_elems,), float("nan"), dtype=out_dtype, device="cuda")
    p.contract(out)
    torch.cuda.synchronize()
    st = p.describe()["steps"][0]
    if tile is not None and torch.cuda.get_device_properties(0).multi_processor_count == 152:
        assert st["tile"] == tile, st
    err = np.abs(out.cpu().numpy().astype(np.float64) - want)
    assert (err <= (4 ** cuts + 8) * 2.0 ** -24 * terms).all(), (err / terms).max() * 2 ** 24
    p.close()
    h.close()


# K = 16 with the default flags: tall results of one or two columns on either
# side of the line between 32 x 32 and 64 x 64 tiles, and 128 x 128 tiles that
# store directly (rows or columns lowest)
@pytest.mark.parametrize("rows,cols,where,tile", [(16, 1, "mixed", SIMT_32x32), (17, 1, "mixed", SIMT_64x64),
                                                  (18, 0, "low", SIMT_64x64), (1, 17, "high", SIMT_64x64),
                                                  (12, 10, "low", SIMT_128x128), (12, 10, "high", SIMT_128x128)])
def test_k16_rules(rows, cols, where, tile):
    n = rows + cols
    first = list(range(rows)) if where == "low" else list(range(cols, n))
    if where == "mixed":
        first = sorted(int(q) for q in np.random.Generator(np.random.PCG64(n)).permutation(n)[:rows])
    rest = [q for q in range(n) if q not in first]
    net = tensors.pseudo_physical_network(n, [(0, 1)] * 2, [first, rest], 5100 + n)
    absnet = Network(n, 2, [Node(nd.out_qubits, nd.cut_ids, nd.cut_role, np.abs(nd.data)) for nd in net.nodes])
    z = oracle.total_mass(net)
    want, terms = oracle.recon_bin_pairwise(net) / z, oracle.recon_bin_pairwise(absnet) / abs(z)
    h = tqc.Network(net)
    p = tqc.Plan(h, precision="fp32")
    out = torch.full((p.out_elems,), float("nan"), dtype=torch.float32, device="cuda")
    p.contract(out)
    torch.cuda.synchronize()
    st = p.describe()["steps"][0]
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        assert st["tile"] == tile, st
    err = np.abs(out.cpu().numpy().astype(np.float64) - want)
    assert (err <= (16 + 8) * 2.0 ** -24 * terms).all(), (err / terms).max() * 2 ** 24
    p.close()
    h.close()
