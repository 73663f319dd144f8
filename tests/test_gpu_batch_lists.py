"""Work lists of the batched launch kept between calls: alternating between
more lists than are kept, plans destroyed in between, and tensors changed
between two launches of a list give what a list built anew gives."""
import numpy as np
import pytest

from gen import tensors

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2502_03445_gb300 import tqc  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def make(seed):
    net = tensors.pseudo_physical_network(14, [(0, 1), (1, 2)], [[0, 3, 6, 9, 12], [1, 4, 7, 10, 13], [2, 5, 8, 11]], seed)
    h = tqc.Network(net)
    p = tqc.Plan(h)
    ref = torch.empty(p.out_elems, dtype=torch.float32, device="cuda")
    p.contract(ref)
    return h, p, ref, torch.empty_like(ref)


def test_alternating_lists():
    """Twelve lists (more than are kept), visited in turn and at random."""
    objs = [make(7000 + i) for i in range(13)]
    rng = np.random.Generator(np.random.PCG64(3))
    for i in list(range(12)) * 2 + [int(x) for x in rng.integers(0, 12, 20)]:
        pair = objs[i:i + 2]
        for _, _, _, out in pair:
            out.zero_()
        tqc.contract_batch([p for _, p, _, _ in pair], [o for _, _, _, o in pair])
        tqc.batch_status()
        for _, _, ref, out in pair:
            assert torch.equal(ref, out)
    for h, p, _, _ in objs:
        p.close()
        h.close()


def test_destroyed_and_changed_plans():
    a, b, c = make(7100), make(7101), make(7102)
    for _ in range(2):
        for lst in ([a, b], [b, c]):
            tqc.contract_batch([x[1] for x in lst], [x[3] for x in lst])
    # a list of a destroyed plan is never found again: a new plan that may
    # sit at the old one's address, with the same output, is its own list
    a[1].close()
    a[0].close()
    tqc.batch_status()
    d = make(7103)
    d[3].zero_()
    tqc.contract_batch([d[1], b[1]], [a[3], b[3]])
    tqc.batch_status()
    assert torch.equal(a[3], d[2]) and torch.equal(b[3], b[2])
    # tensors changed since: refused when the launch moves to another list
    net = tensors.pseudo_physical_network(14, [(0, 1), (1, 2)], [[0, 3, 6, 9, 12], [1, 4, 7, 10, 13], [2, 5, 8, 11]], 7104)
    for j, nd in enumerate(net.nodes):
        c[0].upload(j, nd.data)
    with pytest.raises(tqc.TqcError) as ei:
        tqc.contract_batch([b[1], c[1]], [b[3], c[3]])
    assert ei.value.status == tqc.ERR_INVALID
    c[1].contract(c[2])
    tqc.contract_batch([b[1], c[1]], [b[3], c[3]])
    tqc.batch_status()
    assert torch.equal(c[3], c[2]) and torch.equal(b[3], b[2])
    # the last launched list still reports after its plans are gone
    for h, p, _, _ in (b, c, d):
        p.close()
        h.close()
    tqc.batch_status()


def test_same_list_refused_after_an_upload():
    """The last launched list, launched again: its plans are checked as any
    other's (the cached total mass is that of the tensors before)."""
    a, b = make(7200), make(7201)
    lst = [[x[1] for x in (a, b)], [x[3] for x in (a, b)]]
    for _ in range(2):
        tqc.contract_batch(*lst)
    net = tensors.pseudo_physical_network(14, [(0, 1), (1, 2)], [[0, 3, 6, 9, 12], [1, 4, 7, 10, 13], [2, 5, 8, 11]], 7202)
    for j, nd in enumerate(net.nodes):
        b[0].upload(j, 2 * nd.data)
    with pytest.raises(tqc.TqcError) as ei:
        tqc.contract_batch(*lst)
    assert ei.value.status == tqc.ERR_INVALID
    b[1].contract(b[2])
    tqc.contract_batch(*lst)
    tqc.batch_status()
    assert torch.equal(a[3], a[2]) and torch.equal(b[3], b[2])
    for h, p, _, _ in (a, b):
        p.close()
        h.close()


def test_captured_list_outlives_later_lists():
    """A graph that captured a list is replayed after ten other lists (more
    than are kept) were built."""
    objs = [make(7300 + i) for i in range(12)]
    plans, outs = [o[1] for o in objs[:2]], [o[3] for o in objs[:2]]
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    tqc.contract_batch(plans, outs, stream=s)
    s.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        tqc.contract_batch(plans, outs, stream=s)
    for _, p, ref, out in objs[2:]:
        tqc.contract_batch([p], [out])
        tqc.batch_status()
        assert torch.equal(ref, out)
    for o in outs:
        o.fill_(float("nan"))
    for _ in range(2):
        g.replay()
    torch.cuda.synchronize()
    for _, _, ref, out in objs[:2]:
        assert torch.equal(ref, out)
    del g
    for h, p, _, _ in objs:
        p.close()
        h.close()
