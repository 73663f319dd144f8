"""FP64 results: the FP32 value times the FP64 scale, rounded to nearest even
(formed in integer arithmetic), bit for bit the FP64 product.

P = a (x) [1, 0] without cuts: every value is an entry of a rounded to FP32, the
scale is 1 / Z with Z the sum of a, returned by the call."""
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


def outputs(a, b=(1.0, 0.0), **kw):
    k = int(np.log2(a.size))
    h = tqc.Network(Network(k + 1, 0, [Node(list(range(k)), [], [], a), Node([k], [], [], np.array(b))]))
    p = tqc.Plan(h, **kw)
    out = torch.full((p.out_elems,), float("nan"), dtype=torch.float64, device="cuda")
    z = p.contract(out, want_z=True)
    got = out.cpu().numpy()
    p.close()
    h.close()
    return got[:a.size], got[a.size:], z


def test_ties():
    """The scale is 1 + 2^-30, so an odd 24-bit value's product has 54 bits: a tie."""
    rng = np.random.Generator(np.random.PCG64(1))
    a = (rng.integers(1 << 22, 1 << 23, 1 << 14) * 2 + 1) * rng.choice([-1.0, 1.0], 1 << 14) * 2.0 ** -48
    z = 1.0 / (1.0 + 2.0 ** -30)
    a[-1] = 0.0
    a[-1] = z - a.sum()             # multiples of 2^-53 below 1: every order of the sum is exact
    assert 1.0 / z == 1.0 + 2.0 ** -30
    got, zeros, z_out = outputs(a)
    assert z_out == z and not zeros.any()
    np.testing.assert_array_equal(got, a.astype(np.float32).astype(np.float64) * (1.0 / z))


@pytest.mark.parametrize("seed,exp", [(2, 0), (3, -90), (4, 80)])
def test_any_scale(seed, exp):
    rng = np.random.Generator(np.random.PCG64(seed))
    a = np.ldexp(rng.standard_normal(1 << 14), rng.integers(-30, 10, 1 << 14) + exp)
    a[:64] = np.ldexp(rng.standard_normal(64), -140)     # zero, or subnormal in FP32
    got, _, z = outputs(a)
    np.testing.assert_array_equal(got, a.astype(np.float32).astype(np.float64) * (1.0 / z))


def test_special_values():
    a = np.random.Generator(np.random.PCG64(5)).standard_normal(1 << 14)
    a[:8] = [0.0, np.inf, -np.inf, np.nan, 3.4028234663852886e38, 2.0 ** -149, 2.0 ** -126, 1e300]
    with np.errstate(over="ignore"):
        want = a.astype(np.float32).astype(np.float64)
    got, more, _ = outputs(a, b=(1.0, 1.0), flags=tqc.FLAG_NO_RENORM)
    np.testing.assert_array_equal(got, want)
    np.testing.assert_array_equal(more, want)
