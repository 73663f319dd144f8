"""Ingest: the FP64 -> FP32 conversion, the wide loads' alignment and bin
rules, and the total-mass network, through the public entry points."""
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


def test_fp64_values_are_rounded_to_nearest_fp32():
    """P = a (x) [1, 1] without cuts: every entry is a value of a rounded to
    FP32, ties to even, over normal, subnormal, huge and special values."""
    rng = np.random.Generator(np.random.PCG64(5))
    v = rng.integers(0, 1 << 63, size=1 << 14, dtype=np.uint64).view(np.float64) * rng.choice([-1.0, 1.0], 1 << 14)
    v[:4096] = np.ldexp(rng.integers(1 << 23, 1 << 24, 4096) + 0.5, rng.integers(-170, 110, 4096))    # exact ties
    v[4096:6144] = np.ldexp(rng.random(2048) + 0.5, rng.integers(-152, -120, 2048))                   # subnormals
    v[6144:8192] = np.nextafter(v[:2048], np.inf)                                                     # just above a tie
    v[8192:8200] = [0.0, -0.0, np.inf, -np.inf, np.nan, 3.4028235677973366e38, 3.4028235677973362e38, 2.0 ** -150]
    net = Network(15, 0, [Node(list(range(14)), [], [], v), Node([14], [], [], np.ones(2))])
    h = tqc.Network(net)
    p = tqc.Plan(h, flags=tqc.FLAG_NO_RENORM)
    out = torch.empty(p.out_elems, dtype=torch.float32, device="cuda")
    p.contract(out)
    torch.cuda.synchronize()
    with np.errstate(over="ignore", invalid="ignore"):
        want = v.astype(np.float32)
    got = out.cpu().numpy()
    for half in (got[:1 << 14], got[1 << 14:]):
        np.testing.assert_array_equal(half, want)
    p.close()
    h.close()


# qubits fixed by the bin: source bit 0 or 1 of one subcircuit's tensor or of
# both is then no destination bit, so fewer elements are loaded together
@pytest.mark.parametrize("fixed", [[], [0], [1], [0, 8], [1, 8, 9], [0, 1, 8]])
@pytest.mark.parametrize("dtype", [tqc.F64, tqc.F32])
@pytest.mark.parametrize("prec", ["fp32", "bf16x3", "tf32"])
def test_wide_loads_follow_the_bin(fixed, dtype, prec):
    n = 17
    net = tensors.pseudo_physical_network(n, [(0, 1)] * 3, [list(range(8)), list(range(8, n))], 6000)
    if dtype == tqc.F32:
        net = net.astype(np.float32).astype(np.float64)
    free = [q for q in range(n) if q not in fixed]
    bits = np.ones(n, np.uint8)
    want = oracle.recon_bin_pairwise(net, free, bits) / oracle.total_mass(net)
    h = tqc.Network(net, dtype=dtype)
    p = tqc.Plan(h, precision=prec, free_qubits=free, fixed_bits=bits)
    out = torch.full((p.out_elems,), float("nan"), dtype=torch.float32, device="cuda")
    z = p.contract(out, want_z=True)
    assert abs(z - oracle.total_mass(net)) <= 1e-12
    err = np.abs(out.cpu().numpy().astype(np.float64) - want)
    # FP32-class forms, or (TF32) operands rounded to 11 bits: relative to the terms' size
    assert err.max() <= (1e-5 if prec != "tf32" else 1e-3) * max(np.abs(want).max(), 1.0)
    assert err.sum() <= (1e-4 if prec != "tf32" else 2e-3) * np.abs(want).sum()
    p.close()
    h.close()


@pytest.mark.parametrize("dtype,shift", [(torch.float64, 1), (torch.float32, 1), (torch.float32, 2)])
def test_caller_tensors_of_any_element_alignment(dtype, shift):
    """tqc_contract_noalloc reads the caller's tensors: shifted by `shift`
    elements they are aligned to less than the wide loads need."""
    n = 12
    net = tensors.pseudo_physical_network(n, [(0, 1)] * 2, [list(range(5)), list(range(5, n))], 6100)
    h = tqc.Network(net, shape_only=True)
    p = tqc.Plan(h)
    outs = []
    for k in (0, shift):
        ts = []
        for nd in net.nodes:
            buf = torch.zeros(nd.data.size + 8, dtype=dtype, device="cuda")
            buf[k:k + nd.data.size] = torch.from_numpy(nd.data).to(dtype).cuda()
            ts.append(buf[k:k + nd.data.size])
        out = torch.empty(p.out_elems, dtype=torch.float64, device="cuda")
        p.contract_noalloc(ts, out, in_dtype=tqc.F64 if dtype == torch.float64 else tqc.F32)
        outs.append(out.cpu().numpy())
    np.testing.assert_array_equal(outs[0], outs[1])
    p.close()
    h.close()


# (qubits, cut edges, output counts): one subcircuit, a network whose steps fit
# one cluster, one with more than 2^18 multiply-adds (a launch per step)
MASS = [(3, [], [3]), (12, [(0, 1)] * 2 + [(1, 2)], [4, 4, 4]), (9, [(0, 1)] * 4 + [(1, 2)] * 4 + [(0, 2)] * 3, [3, 3, 3])]


@pytest.mark.parametrize("n,edges,counts", MASS)
@pytest.mark.parametrize("sliced", [[], [0]])
def test_total_mass(n, edges, counts, sliced):
    """Z against the FP64 oracle (Gaussian tensors: sums that cancel), within
    the rounding of any order of its terms."""
    if sliced and not edges:
        pytest.skip("no cut to slice")
    outs, at = [], 0
    for c in counts:
        outs.append(list(range(at, at + c)))
        at += c
    rng = np.random.Generator(np.random.PCG64(n))
    nodes = []
    for j, o in enumerate(outs):
        cuts = [(c, e.index(j)) for c, e in enumerate(edges) if j in e]
        nodes.append(Node(o, [c for c, _ in cuts], [r for _, r in cuts], rng.standard_normal((4 ** len(cuts)) << len(o))))
    net = Network(n, len(edges), nodes)
    net.check()
    absnet = Network(n, len(edges), [Node(d.out_qubits, d.cut_ids, d.cut_role, np.abs(d.data)) for d in nodes])
    h = tqc.Network(net)
    p = tqc.Plan(h, flags=tqc.FLAG_NO_RENORM, sliced=sliced)
    out = torch.empty(p.out_elems, dtype=torch.float32, device="cuda")
    z = p.contract(out, want_z=True)
    steps = sum(4 ** len(d.cut_ids) << len(d.out_qubits) for d in nodes) + 4 ** len(edges)
    assert abs(z - oracle.total_mass(net)) <= 2 * np.log2(steps) * 2.0 ** -52 * oracle.total_mass(absnet) * len(nodes) * 8
    p.close()
    h.close()


def test_total_mass_of_a_leaf_with_13_cuts():
    """2^26 destinations of a summed leaf: 2^31 threads wanted, more than 32
    bits hold, must still give the launch its whole grid and not one CTA
    (about 2^23 dependent rounds of a warp, seconds; the whole contract moves
    2 GB, a few milliseconds)."""
    edges = [(0, 1)] * 5 + [(0, 2)] * 4 + [(0, 3)] * 4
    outs = [[0], [1, 2], [3, 4], [5]]
    rng = np.random.Generator(np.random.PCG64(26))
    nodes = []
    for j, o in enumerate(outs):
        cuts = [(c, e.index(j)) for c, e in enumerate(edges) if j in e]
        nodes.append(Node(o, [c for c, _ in cuts], [r for _, r in cuts],
                          rng.random((4 ** len(cuts)) << len(o), dtype=np.float32)))
    t = [d.data.reshape(-1, 1 << len(d.out_qubits)).sum(1, dtype=np.float64) for d in nodes]
    want = ((t[0].reshape(-1, 4 ** 4) @ t[3]).reshape(4 ** 5, 4 ** 4) @ t[2]) @ t[1] / 2 ** len(edges)
    h = tqc.Network(Network(6, len(edges), nodes), dtype=tqc.F32)
    p = tqc.Plan(h)
    out = torch.empty(p.out_elems, dtype=torch.float32, device="cuda")
    p.contract(out)
    h.upload(3, nodes[3].data)  # the next call computes the mass again
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record()
    p.contract(out)
    e1.record()
    e1.synchronize()
    z = p.contract(out, want_z=True)
    assert abs(z - want) <= 1e-12 * want  # positive terms
    assert e0.elapsed_time(e1) < 500, e0.elapsed_time(e1)
    p.close()
    h.close()
