"""The elements of a row past its cells: steps store whole sectors and write some
of them.  An adjoint field's padding stays zero, so that sums over the field's
buffer are sums over its cells; no result depends on what the padding holds."""
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


@pytest.mark.parametrize("Q", [27, 15])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("walls", [0, 3])
@pytest.mark.parametrize("shape", [(3, 4, n) for n in (1, 2, 7, 9, 30, 33, 257)]
                         + [(20, 41, 33)])  # the last: odd rows on the two-cell kernel
def test_adjoint_fields_keep_zero_padding(lbm, Q, storage, walls, shape):
    """From lam_next with a poisoned padding to lam_out with a zero one: zero
    still, and the cells as from lam_next without the poison."""
    om = W.omegas(Q, 1 / 0.6)
    lam = torch.as_tensor(W.rng(5).standard_normal((Q,) + shape))
    F = W.rng(6).uniform(-1e-3, 1e-3, (3,) + shape)
    got = []
    for fill in (0.0, float("nan")):
        S = lbm.Solver(Q, shape, om, walls=walls, force=F, storage=storage)
        S.set_state(W.random_field_state(shape, Q, spread=0.2))
        a, b = S.new_adjoint_field(), S.new_adjoint_field()
        a.fill_(fill)
        S.adjoint_view(a).copy_(lam)
        gF = torch.zeros((3,) + shape, dtype=torch.float32, device="cuda")
        S.adjoint_step(S.current_buffer(), a, b, gF)
        padding = b.view((Q,) + shape[:2] + (lbm.lbm_row_pitch(S.ctx),))[..., shape[2]:]
        assert torch.equal(padding, torch.zeros_like(padding))
        got.append((S.adjoint_view(b).clone(), gF))
    assert torch.isfinite(got[0][0]).all()
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
