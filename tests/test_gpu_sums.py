"""Global sums of grids with more groups of rows than the reductions launch blocks
(1,216), so that a block takes a second group.  A cell's moments are FP32 sums of
its Q stored deviations (and half its force), each of the at most Q + 1 roundings
off by at most 2^-24 of the sum of their magnitudes; the sums over cells are FP64.
The state is biased, so that a row lost or taken twice is far outside that."""
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


@pytest.mark.parametrize("Q", [27, 15])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("inplace", [False, True])
@pytest.mark.parametrize("shape", [(50, 51, 34), (36, 36, 100)])  # 1,275 and 1,296 groups
def test_sums_of_many_rows(lbm, Q, storage, inplace, shape):
    F = np.array([1e-3, 2e-3, 5e-4])
    bias = np.array([0.02, 0.03, 0.04])
    e = oracle.lattice(Q)[0]
    w = oracle.equilibrium(Q, np.ones((1, 1, 1)), np.zeros((3, 1, 1, 1)), np.zeros(3))
    S = lbm.Solver(Q, shape, W.omegas(Q, 1 / 0.6), force=F, walls=2, storage=storage,
                   inplace=inplace)
    S.set_state(w * (1.05 + 3 * (e @ bias).reshape(Q, 1, 1, 1)
                     + 0.02 * W.rng(21).uniform(-1, 1, (Q,) + shape)))
    f = S.get_state().cpu().numpy()
    dev, half = f - w, F.reshape(3, 1, 1, 1) / 2
    drho = dev.sum(0)
    j = np.tensordot(e.T, dev, 1) + half
    want = np.r_[drho.sum(), j.sum((1, 2, 3))]
    cell = (Q + 1) * 2.0 ** -24 * (np.abs(dev).sum(0) + np.abs(half).max())  # of a moment
    row = np.abs(np.stack([drho, *j]).sum(-1)).min((1, 2))
    assert (row > 10 * cell.sum()).all()
    got = S.conservation()
    N = drho.size
    np.testing.assert_allclose(got - [N, 0, 0, 0], want, rtol=0, atol=cell.sum())
    out = torch.full((4,), float("nan"), dtype=torch.float64, device="cuda")
    lbm.lbm_conservation_noalloc(S.ctx, out)
    np.testing.assert_array_equal(out.cpu().numpy() + [N, 0, 0, 0], got)
    # |j|^2 / (2 rho): the moments' errors, and 10 roundings of the value
    energy = 0.5 * (j * j).sum(0) / (1 + drho)
    atol = ((np.abs(j).sum(0) + energy) * cell + 10 * 2.0 ** -24 * energy).sum()
    assert energy.sum(-1).min() > 10 * atol
    np.testing.assert_allclose(S.kinetic_energy(), energy.sum(), rtol=0, atol=atol)
