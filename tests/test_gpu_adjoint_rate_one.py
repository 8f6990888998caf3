"""The adjoint step of D3Q27 where the rates from the trace on are all 1 (its own
form of the kernel): against the FP64 oracle's complex-step adjoint, and against
the general form, forced by the float below 1 as the last rate.  Bound: 1e-5 of
the largest value, FP32 arithmetic of ~10^3 operations per cell on O(1) adjoints;
the other form differs from it in ~100 operations and in that rate, 2e-6."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("walls", [0, 1, 3])
@pytest.mark.parametrize("shape", [(1, 1, 2), (4, 5, 3), (3, 4, 8), (2, 3, 72), (2, 2, 257)])
def test_rate_one_adjoint(lbm, storage, walls, shape):
    import oracle
    Q = 27
    F = W.rng(5).uniform(-1e-2, 1e-2, (3,) + shape).astype(np.float32).astype(np.float64)
    lam = W.rng(6).standard_normal((Q,) + shape).astype(np.float32).astype(np.float64)
    got = []
    for last in (1.0, np.nextafter(np.float32(1.0), np.float32(0.0))):
        om = W.omegas(Q, 1 / 0.6)
        om[26] = last
        S = lbm.Solver(Q, shape, om, force=F, walls=walls, storage=storage)
        S.set_state(W.random_field_state(shape, Q, spread=0.3))
        a, b = S.new_adjoint_field(), S.new_adjoint_field()
        S.adjoint_view(a).copy_(torch.as_tensor(lam))
        gF = torch.zeros((3,) + shape, dtype=torch.float32, device="cuda")
        S.adjoint_step(S.current_buffer(), a, b, gF)
        got.append((S.adjoint_view(b).cpu().numpy(), gF.cpu().numpy()))
        f = S.get_state().cpu().numpy()
    want_F = np.zeros((3,) + shape)
    want = oracle.adjoint_step(Q, shape, f, F, W.omegas(Q, 1 / 0.6), lam, bc=walls, gF=want_F)
    for k, exact in ((0, want), (1, want_F)):
        big = np.abs(exact).max()
        np.testing.assert_allclose(got[0][k], exact, rtol=0, atol=1e-5 * big)
        np.testing.assert_allclose(got[0][k], got[1][k], rtol=0, atol=2e-6 * big)
