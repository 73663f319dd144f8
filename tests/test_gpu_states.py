"""Arbitrary state lists (tqc_contract_states) against the FP64 oracles.

§VII-C reconstructs lists of arbitrary states.  Each state's probability is
checked element by element: oracle A (brute force over every cut
assignment) on the 30-qubit grid network and small networks, oracle B
(per-state elimination, spawned processes) on the 48-qubit QAOA bin network.

Gates: the fused form computes in FP32 on CUDA cores, so it meets the FP32
gate (1e-5 absolute per probability, and 1e-4 of the largest one).  The
per-state form runs the plan's own step kernels: the same FP32-class gate
when its tensor-core steps are split BF16, the 1e-3 total-variation gate
(over the listed states) when one is TF32."""
import numpy as np
import pytest

import oracle
from gen import Network, Node, tensors, workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2502_03445_gb300 import tqc  # noqa: E402

FP32_ATOL = 1e-5
TC_TV = 1e-3


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def states_of(n_qubits, count, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    return rng.integers(0, 1 << n_qubits, size=count, dtype=np.uint64)


def run_states(h, states, out_dtype=torch.float32, **kw):
    p = tqc.Plan(h, free_qubits=[], **kw)
    out = torch.full((len(states),), float("nan"), dtype=out_dtype, device="cuda")
    z = p.contract_states(states, out, want_z=True)
    torch.cuda.synchronize()
    d = p.describe()
    p.close()
    return out.cpu().numpy().astype(np.float64), z, d


def check_fp32(got, want):
    err = np.abs(got - want).max()
    assert err <= FP32_ATOL, err
    assert err <= 1e-4 * np.abs(want).max(), (err, np.abs(want).max())


def test_grid30_ten_thousand_states():
    """The 30-qubit grid network: 10^4 uniformly drawn states, fused form."""
    net = workloads.grid30(0)
    st = states_of(30, 10_000, 31)
    h = tqc.Network(net)
    got, z, d = run_states(h, st)
    assert d["states_form"] == "fused"
    z_or = oracle.total_mass(net)
    assert abs(z - z_or) <= 1e-9
    want = oracle.recon_states(net, st) / z_or
    check_fp32(got, want)
    # the same states through the full 2^30 bin
    p = tqc.Plan(h)
    full = torch.empty(p.out_elems, dtype=torch.float32, device="cuda")
    p.contract(full)
    fb = full[torch.from_numpy(st.astype(np.int64)).cuda()].double().cpu().numpy()
    assert np.abs(fb - got).max() <= 2 * FP32_ATOL
    p.close()
    h.close()


SMALL = [(13, 2, 4, 10), (14, 3, 5, 10), (15, 4, 7, 10), (16, 3, 8, 12), (14, 5, 8, 10), (16, 6, 9, 10)]


@pytest.mark.parametrize("seed", range(len(SMALL)))
def test_small_networks_fused(seed):
    """Shape-matched networks of 2-6 subcircuits (n, m, cuts, width as
    listed), with repeated states and FP64 output."""
    net = tensors.shape_matched_network(*SMALL[seed], seed=3700 + seed)
    st = states_of(net.n_qubits, 700, seed)
    st[::7] = st[0]                                  # duplicates
    h = tqc.Network(net)
    for out_dtype in (torch.float32, torch.float64):
        got, z, d = run_states(h, st, out_dtype)
        assert d["states_form"] == "fused"
        check_fp32(got, oracle.recon_states(net, st) / oracle.total_mass(net))
    h.close()


def test_zero_cuts_single_subcircuit_and_empty_list():
    rng = np.random.Generator(np.random.PCG64(8))
    a, b = rng.random(8), rng.random(16)
    outer = Network(7, 0, [Node([5, 0, 2], [], [], a / a.sum()), Node([1, 3, 6, 4], [], [], b / b.sum())])
    one = Network(5, 0, [Node([4, 0, 2, 1, 3], [], [], rng.random(32))])
    for net in (outer, one):
        net.check()
        st = states_of(net.n_qubits, 100, 9)
        h = tqc.Network(net)
        got, z, d = run_states(h, st)
        assert d["states_form"] == "fused"
        check_fp32(got, oracle.recon_states(net, st) / oracle.total_mass(net))
        p = tqc.Plan(h, free_qubits=[])
        p.contract_states(np.zeros(0, np.uint64), torch.empty(0, device="cuda"))
        p.close()
        h.close()


def test_no_renorm_and_uploads():
    """Raw probabilities with TQC_FLAG_NO_RENORM; new tensors are seen (the
    per-node tables are rebuilt when the tensors change)."""
    base = tensors.shape_matched_network(12, 3, 5, 9, seed=3800)
    nets = [tensors.random_data_network(base, s) for s in (1, 2)]
    st = states_of(12, 500, 3)
    h = tqc.Network(nets[0])
    p = tqc.Plan(h, free_qubits=[], flags=tqc.FLAG_NO_RENORM)
    out = torch.empty(len(st), dtype=torch.float64, device="cuda")
    for k, net in enumerate(nets):
        if k:
            for j, nd in enumerate(net.nodes):
                h.upload(j, nd.data)
        z = p.contract_states(st, out, want_z=True)
        torch.cuda.synchronize()
        want = oracle.recon_states(net, st)
        assert abs(z - oracle.total_mass(net)) <= 1e-9 * abs(oracle.total_mass(net))
        err = np.abs(out.cpu().numpy() - want).max()
        assert err <= 1e-4 * np.abs(want).max(), err
    p.close()
    h.close()


def test_qaoa48_per_state_form():
    """The 48-qubit QAOA bin network: single-state intermediates of 4^12
    floats run per state through the step kernels; 1024 uniformly drawn
    states against oracle B."""
    net = workloads.qaoa48(0)
    st = states_of(net.n_qubits, 1024, 48)
    h = tqc.Network(net)
    p = tqc.Plan(h, free_qubits=[])
    d = p.describe()
    assert d["states_form"] == "per-state"
    out = torch.empty(len(st), dtype=torch.float32, device="cuda")
    z = p.contract_states(st, out, want_z=True)
    torch.cuda.synchronize()
    got = out.cpu().numpy().astype(np.float64)
    want = oracle.recon_states_elim_pool(("gen.workloads", "qaoa48", (0,)), [int(s) for s in st]) / z
    assert abs(z - oracle.total_mass(net)) <= 1e-9 * abs(z)
    err = np.abs(got - want)
    tv = 0.5 * err.sum() / np.abs(want).sum()
    print(f"qaoa48 states: steps {[(s['log2_m'], s['log2_n'], s['log2_k'], s['class'], s['prec']) for s in d['steps']]}"
          f" max|err| {err.max():.3e} max|P| {np.abs(want).max():.3e} tv {tv:.3e}")
    assert err.max() <= FP32_ATOL
    if any(s["class"] == "tcgen05" and s["prec"] == "tf32" for s in d["steps"]):
        assert tv <= TC_TV
    else:
        # FP32-class steps summing up to 4^8 signed terms: within n_steps * 2^-12
        # of the mean absolute term mass per state (the reconstruction with
        # |T_j| in place of T_j, over 2^n), as for the full-size bins
        a = Network(net.n_qubits, net.n_cuts,
                    [Node(nd.out_qubits, nd.cut_ids, nd.cut_role, np.abs(nd.data)) for nd in net.nodes])
        scale = oracle.total_mass(a) / float(1 << net.n_qubits) / abs(z)
        assert err.max() <= max(1e-4 * np.abs(want).max(), len(d["steps"]) * 2.0 ** -12 * scale), (err.max(), scale)
    p.close()
    h.close()


def test_rejections():
    net = tensors.shape_matched_network(12, 3, 5, 9, seed=3900)
    h = tqc.Network(net)
    out = torch.empty(4, dtype=torch.float32, device="cuda")
    p = tqc.Plan(h)                                     # free qubits: not a single-state plan
    with pytest.raises(tqc.TqcError) as ei:
        p.contract_states([1, 2, 3, 4], out)
    assert ei.value.status == tqc.ERR_INVALID
    p.close()
    p = tqc.Plan(h, free_qubits=[], sliced=[1])
    with pytest.raises(tqc.TqcError) as ei:
        p.contract_states([1, 2, 3, 4], out)
    assert ei.value.status == tqc.ERR_UNSUPPORTED
    p.close()
    p = tqc.Plan(h, free_qubits=[])
    with pytest.raises(tqc.TqcError) as ei:
        p.contract_states([1, 2, 3, 1 << 12], out)      # a bit beyond n_qubits
    assert ei.value.status == tqc.ERR_INVALID
    p.close()
    h.close()


# Three subcircuits joined pairwise by 3, 2 and 1 cuts (the first pair's step,
# 64 x .. x 64, is worth sharing between states), a chain of four (every step
# small), and a ring whose last subcircuit has no outputs.
SPLITS = {
    "triangle": (14, [(0, 1)] * 3 + [(1, 2)] * 2 + [(0, 2)], [[0, 5, 9], [1, 4, 8, 11], [2, 3, 6, 7, 10, 12, 13]]),
    "chain": (13, [(0, 1), (1, 2), (2, 3)], [[3, 7, 8], [0, 1, 12], [2, 5, 6, 11], [4, 9, 10]]),
    "ring": (12, [(0, 1), (1, 2), (2, 3), (0, 3), (0, 2)], [[0, 3, 6, 9], [1, 4, 7, 10], [2, 5, 8, 11], []]),
}


@pytest.mark.parametrize("name", list(SPLITS))
@pytest.mark.parametrize("count", [1, 31, 257, 5000, 70001])
def test_list_lengths_and_orders(name, count):
    """Lists from one state to more than the states there are: random,
    descending, and one state repeated, each state against the whole
    distribution by the FP64 oracle."""
    n, edges, outs = SPLITS[name]
    net = tensors.pseudo_physical_network(n, edges, outs, 4000 + count)
    want = oracle.recon_bin(net) / oracle.total_mass(net)
    h = tqc.Network(net)
    for st in (states_of(n, count, count), np.sort(states_of(n, count, 1 + count))[::-1].copy(),
               np.full(count, (1 << n) - 2, np.uint64)):
        got, z, d = run_states(h, st)
        assert d["states_form"] == "fused"
        check_fp32(got, want[st.astype(np.int64)])
    h.close()


# More networks, for which other splits of the steps are the fastest or the
# only ones that fit: a step of 2^18 multiply-adds with an operand larger than
# shared memory, and one (seven subcircuits) whose leaf operands only fit in
# turn.  Entries are positive: sums of up to 2^38 terms do not cancel.
MORE = {
    "heavy": (10, [(0, 1), (1, 2), (1, 3), (2, 1), (1, 0), (1, 2), (1, 3), (1, 0), (1, 2)],
              [[2, 3, 5], [0, 1, 6, 7, 9], [4], [8]]),
    "in_turn": (7, [(0, 1), (0, 2), (2, 3), (2, 4), (4, 5), (2, 6), (1, 0), (6, 2), (6, 0), (2, 4), (1, 4), (0, 5), (3, 2),
                    (6, 3), (6, 0), (5, 4), (4, 5), (6, 4), (1, 0)], [[4, 5], [], [6], [3], [2, 0], [], [1]]),
}


@pytest.mark.parametrize("name", list(SPLITS) + list(MORE))
def test_a_state_has_one_fp64_value_in_every_list(name):
    """Lists of 1 to 10^6 states (other splits of the steps; at 10^6 a CTA's
    window of the sorted list moves, and with one state repeated a group is
    longer than a CTA's threads): FP64 results bit for bit those of the list of
    all states, FP32 ones within the FP32 gate."""
    n, edges, outs = {**SPLITS, **MORE}[name]
    net = tensors.pseudo_physical_network(n, edges, outs, 4100)
    if name in MORE:
        net = Network(n, net.n_cuts, [Node(d.out_qubits, d.cut_ids, d.cut_role, np.abs(d.data)) for d in net.nodes])
    want = oracle.recon_bin_pairwise(net) / oracle.total_mass(net)
    h = tqc.Network(net)
    every, _, d = run_states(h, np.arange(1 << n, dtype=np.uint64), torch.float64)
    assert d["states_form"] == "fused"
    check_fp32(every, want)
    lists = [np.full(1, x, np.uint64) for x in (0, (1 << n) - 1, 37)]
    lists += [states_of(n, c, c) for c in (40, 300, 2000, 40_000, 1_000_000)] + [np.full(1_000_000, 21, np.uint64)]
    for st in lists:
        got, _, _ = run_states(h, st, torch.float64)
        np.testing.assert_array_equal(got, every[st.astype(np.int64)])
        got, _, _ = run_states(h, st)
        check_fp32(got, want[st.astype(np.int64)])
    h.close()


def test_a_short_list_takes_little_memory():
    """1000 states of 26 qubits: the plan's tables (2 MB) and tens of bytes per
    state, not a counter for every value of the sort key (2^22 of them)."""
    net = tensors.shape_matched_network(26, 4, 6, 12, seed=4200)
    h = tqc.Network(net)
    st = states_of(26, 1000, 1)
    out = torch.empty(len(st), dtype=torch.float32, device="cuda")
    warm = tqc.Plan(h, free_qubits=[])           # the kernels are loaded
    warm.contract_states(st, out)
    p = tqc.Plan(h, free_qubits=[])
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    p.contract_states(st, out)
    torch.cuda.synchronize()
    used = before - torch.cuda.mem_get_info()[0]
    tables = sum(4 * nd.data.size for nd in net.nodes)
    assert used <= tables + (8 << 20), (used, tables)
    check_fp32(out.cpu().numpy().astype(np.float64), oracle.recon_states(net, st) / oracle.total_mass(net))
    for q in (p, warm):
        q.close()
    h.close()
