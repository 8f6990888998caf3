"""Loading and reading a state, and the global sums.

FP32 storage: set_state stores float(f - w) and get_state returns
w + double(stored), both correctly rounded, so the round trip is known bit for
bit for every input, ordinary or not.  The sums are compared with FP64 sums of
the state read back; a cell's moments are FP32 sums of Q deviations of at most
m in size, so each sum is off by at most N Q^2 2^-24 m."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def lbm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1202_6081_gb300 import build
    from paper_1202_6081_gb300 import lbm as mod
    build()
    mod.load()
    return mod


def _weights(Q):
    # the oracle's rest state: f^at(rho = 1, u = 0)
    one = (1, 1, 1)
    f = oracle.equilibrium(Q, np.ones(one), np.zeros((3,) + one), np.zeros(3)).reshape(Q)
    n = (oracle.lattice(Q)[0] ** 2).sum(1)
    table = ({0: 8 / 27, 1: 2 / 27, 2: 1 / 54, 3: 1 / 216} if Q == 27 else
             {0: 2 / 9, 1: 1 / 9, 3: 1 / 72})
    w = np.array([table[int(k)] for k in n])
    np.testing.assert_allclose(f, w, rtol=1e-14)
    return w


@pytest.mark.parametrize("Q", [27, 15])
@pytest.mark.parametrize("walls,inplace", [(0, False), (3, False), (0, True), (2, True)])
@pytest.mark.parametrize("spread", [0.0, 1e-13, 1e-9, 1e-4, 0.4, 3.0, 1e30])
def test_fp32_round_trip_is_exactly_rounded(lbm, Q, walls, inplace, spread):
    shape = (3, 5, 34)
    w = _weights(Q).reshape(Q, 1, 1, 1)
    f = w * (1 + spread * W.rng(11).uniform(-1, 1, (Q,) + shape))
    f[:, 0, 0, 0] = w[:, 0, 0, 0]
    f[:, 0, 0, 1] = np.nextafter(w[:, 0, 0, 0], 0)
    f[:, 0, 0, 2] = 2 * w[:, 0, 0, 0]
    f[:, 0, 0, 3] = w[:, 0, 0, 0] / 2
    f[:, 0, 0, 4] = 0.0
    f[:, 0, 0, 5] = np.inf
    f[:, 0, 0, 6] = np.nan
    S = lbm.Solver(Q, shape, W.omegas(Q, 1 / 0.6), walls=walls, inplace=inplace)
    S.set_state(f)
    got = S.get_state().cpu().numpy()
    want = w + (f - w).astype(np.float32).astype(np.float64)
    np.testing.assert_array_equal(got, want)


# rows of one to several blocks' width, short rows sharing a block, and more
# groups of rows than blocks
SHAPES = [(1, 1, 1), (3, 5, 3), (2, 7, 17), (4, 3, 90), (2, 3, 129), (2, 2, 300), (40, 41, 33)]


@pytest.mark.parametrize("Q", [27, 15])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("shape", SHAPES)
def test_sums_match_the_state_read_back(lbm, Q, storage, shape):
    F = np.array([1e-3, -2e-3, 5e-4])
    S = lbm.Solver(Q, shape, W.omegas(Q, 1 / 0.6), force=F, walls=2, storage=storage)
    S.set_state(W.random_field_state(shape, Q))
    f = S.get_state().cpu().numpy()
    N, e = int(np.prod(shape)), oracle.lattice(Q)[0]
    j = np.tensordot(e.T, f, 1) + F.reshape(3, 1, 1, 1) / 2
    rho = f.sum(0)
    bound = N * Q * Q * 2.0 ** -24
    np.testing.assert_allclose(S.conservation(), np.r_[rho.sum(), j.sum((1, 2, 3))], rtol=0,
                               atol=bound)
    out = torch.full((4,), float("nan"), dtype=torch.float64, device="cuda")
    lbm.lbm_conservation_noalloc(S.ctx, out)
    np.testing.assert_array_equal(out.cpu().numpy() + [N, 0, 0, 0], S.conservation())
    # the energy is quadratic in moments below 2: twice their bound, times 3 axes
    np.testing.assert_allclose(S.kinetic_energy(), 0.5 * ((j * j).sum(0) / rho).sum(), rtol=0,
                               atol=6 * bound)
