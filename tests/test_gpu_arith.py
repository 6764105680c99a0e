"""The recurrent kernels' scalar arithmetic against IEEE divides, through qnn_selftest_pair_functions:
the reciprocal from the hardware approximation and one Newton step is correctly rounded for every
significand (checked at exponents across its range; scaling by a power of two changes no rounding
while nothing leaves the normal range), and sigma, tanh and the cell update equal their clamped,
divided forms on both sides of the argument limit that separates them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qnn():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1607_04683_gb300 import build, qnn as q
    build.build()
    q.lib()
    torch.cuda.set_device(0)
    return q


@pytest.mark.parametrize("exponent", [-100, -61, -60, -1, 0, 1, 6, 60, 61, 124, 125])
def test_reciprocal_every_significand(qnn, exponent):
    bits = torch.arange(1 << 23, dtype=torch.int32, device="cuda") + ((exponent + 127) << 23)
    assert qnn.selftest_pair_functions(bits.view(torch.float32)) == 0


def test_activations_around_the_argument_limit(qnn):
    g = np.random.Generator(np.random.PCG64(5))
    lim = np.float32(86.0)
    edge = np.array([0.0, -0.0, lim, lim / 2, 87.0, 88.0, 43.5, 44.0, np.inf, 1e-30, 3e38], np.float32)
    edge = np.concatenate([edge, np.nextafter(edge, np.float32(0)), np.nextafter(edge, np.float32(np.inf))])
    edge = np.concatenate([edge, -edge])
    pairs = np.stack(np.meshgrid(edge, edge), -1).reshape(-1)
    rnd = g.uniform(-100, 100, 1 << 20) * np.exp2(-g.integers(0, 20, 1 << 20).astype(np.float64))
    for v in (pairs, rnd):
        assert qnn.selftest_pair_functions(torch.from_numpy(v.astype(np.float32)).cuda()) == 0
