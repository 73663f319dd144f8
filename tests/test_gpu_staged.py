"""Staged write-out of tensor-core steps: every arrangement of the result's
lowest bits over rows and columns, whole and partial sub-tiles, every output
form, against the FP64 oracle.

Bound (split BF16): operands carry 17 bits (relative error 2^-17 each), the
lo * lo product dropped is at most 2^-16 of a term, and K additions round at
2^-23: |error| <= (2^-14 + K 2^-23) sum_k |a_k| |b_k|, the sum being the
oracle's value on absolute tensors.  TF32: 11-bit operands, 2^-10 in all."""
import numpy as np
import pytest

import oracle
from gen import Network, Node, tensors

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2502_03445_gb300 import tqc  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


# the row qubits among the lowest ones; the others are columns
PATTERNS = {"rows01": [0, 1, 4, 6, 9], "cols01": [2, 3, 5, 8, 10], "row_col": [0, 2, 3, 7, 11], "col_row": [1, 3, 4, 6, 12],
            "far": [0, 9, 11, 13, 14], "alternate": [0, 2, 4, 6, 8, 10, 12, 14], "blocks": [1, 2, 5, 6, 9, 10, 13]}


def check(net, n, out, scale_bound):
    absnet = Network(n, net.n_cuts, [Node(d.out_qubits, d.cut_ids, d.cut_role, np.abs(d.data)) for d in net.nodes])
    z = oracle.total_mass(net)
    want, terms = oracle.recon_bin_pairwise(net) / z, oracle.recon_bin_pairwise(absnet) / abs(z)
    err = np.abs(out.cpu().numpy().astype(np.float64) - want)
    assert (err <= scale_bound * terms).all(), (err / terms).max() / scale_bound


@pytest.mark.parametrize("pat", sorted(PATTERNS))
@pytest.mark.parametrize("rows,cols", [(9, 8), (8, 5), (9, 5), (12, 4), (11, 7), (6, 10)])
@pytest.mark.parametrize("prec,dtype", [("bf16x3", torch.float32), ("bf16x3", torch.float64), ("tf32", torch.float32)])
def test_final_step(pat, rows, cols, prec, dtype):
    n = rows + cols
    first = [q for q in PATTERNS[pat] if q < n][:rows]
    rest = [q for q in range(n) if q not in first]
    rng = np.random.Generator(np.random.PCG64(rows * 100 + cols))
    first = sorted(first + [int(q) for q in rng.permutation([q for q in rest if q > 4])[:rows - len(first)]])
    if len(first) < rows:  # not enough qubits above the pattern's low ones
        first = sorted(first + [q for q in rest if q not in first][:rows - len(first)])
    rest = [q for q in range(n) if q not in first]
    net = tensors.pseudo_physical_network(n, [(0, 1)] * 3, [first, rest], 8000 + n)
    h = tqc.Network(net)
    p = tqc.Plan(h, precision=prec)
    out = torch.full((p.out_elems,), float("nan"), dtype=dtype, device="cuda")
    p.contract(out)
    torch.cuda.synchronize()
    assert p.describe()["steps"][0]["class"] == ("tcgen05" if n >= 14 else "simt")
    check(net, n, out, 2.0 ** -14 + 64 * 2.0 ** -23 if prec == "bf16x3" else 2.0 ** -9)
    p.close()
    h.close()


@pytest.mark.parametrize("pat", sorted(PATTERNS))
@pytest.mark.parametrize("sliced", [[], [0]])
def test_intermediate_and_sliced_steps(pat, sliced):
    """Split-BF16, TF32-free operands of a second tensor-core step, and the
    FP64 slice sum."""
    n = 18
    first = PATTERNS[pat][:6]
    others = [q for q in range(n) if q not in first]
    net = tensors.pseudo_physical_network(n, [(0, 1)] * 4 + [(1, 2)] * 3, [first, others[0::2], others[1::2]], 8100)
    h = tqc.Network(net)
    p = tqc.Plan(h, precision="bf16x3", order=[[0, 1], [3, 2]], sliced=sliced)
    out = torch.full((p.out_elems,), float("nan"), dtype=torch.float32, device="cuda")
    p.contract(out)
    torch.cuda.synchronize()
    check(net, n, out, 2 * (2.0 ** -14 + 256 * 2.0 ** -23))
    p.close()
    h.close()


@pytest.mark.parametrize("pat", ["rows01", "cols01", "row_col", "col_row"])
@pytest.mark.parametrize("prec", ["bf16x3", "tf32", "bf16"])
def test_wide_tiles(pat, prec):
    """128 x 256 staged tiles (K = 256, a tile for every SM); split BF16 takes
    64-byte k-blocks there."""
    n = 23
    first = PATTERNS[pat]
    first = sorted(first + [q for q in range(13, 21)])
    rest = [q for q in range(n) if q not in first]
    net = tensors.pseudo_physical_network(n, [(0, 1)] * 4, [first, rest], 8200)
    h = tqc.Network(net)
    p = tqc.Plan(h, precision=prec)
    out = torch.full((p.out_elems,), float("nan"), dtype=torch.float32, device="cuda")
    p.contract(out)
    torch.cuda.synchronize()
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        assert p.describe()["steps"][0]["tile"] in (3, 4)  # 3: stores that fill whole sectors
    # BF16: 8-bit operands, 2^-7 in all
    check(net, n, out, {"bf16x3": 2.0 ** -14 + 256 * 2.0 ** -23, "tf32": 2.0 ** -9, "bf16": 2.0 ** -7}[prec])
    p.close()
    h.close()
