"""Rows of odd length on grids above the size that the one-cell kernels serve (16
warps on an SM): the two-cell kernels, whose last thread of a row has one cell and
whose threads past it store in the padding."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SHAPES = [(20, 21, 257), (30, 41, 41)]  # 27 and 20 warps


@pytest.fixture(scope="module")
def lbm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1202_6081_gb300 import build
    from paper_1202_6081_gb300 import lbm as mod
    build()
    mod.load()
    return mod


def _solver(lbm, Q, shape, walls, form, **kw):
    """form: D3Q27 the rate-1 relaxation, D3Q15 a force (a field)."""
    om = W.omegas(Q, 1 / 0.6) if Q == 27 and form else W.random_omegas(Q, seed=12)
    F = np.asarray(W.rng(13).uniform(-2e-3, 2e-3, (3,) + shape), dtype=np.float32)
    if Q == 15 and not form:
        F = np.zeros(3)
    return lbm.Solver(Q, shape, om, walls=walls, force=F, **kw), om, F.astype(np.float64)


@pytest.mark.parametrize("Q", [27, 15])
@pytest.mark.parametrize("walls", [0, 3])
@pytest.mark.parametrize("form", [False, True])
@pytest.mark.parametrize("shape", SHAPES)
def test_step_matches_oracle(lbm, Q, walls, form, shape):
    """One step against the FP64 oracle, at the bound of the other FP32 steps (from
    this state the D3Q27 flow has no positive density after three)."""
    import oracle
    f = W.random_field_state(shape, Q, seed=14, spread=0.5)
    S, om, F = _solver(lbm, Q, shape, walls, form)
    S.set_state(f)
    S.step(1)
    want = oracle.run(Q, shape, f, F, om, 1, bc=walls)
    assert np.abs(S.get_state().cpu().numpy() - want).max() <= 2e-6


@pytest.mark.parametrize("Q", [27, 15])
@pytest.mark.parametrize("walls", [0, 3])
@pytest.mark.parametrize("shape", SHAPES)
def test_results_do_not_depend_on_the_padding(lbm, Q, walls, shape):
    out = []
    for fill in (0x00, 0xff):  # zeros, NaNs
        S = _solver(lbm, Q, shape, walls, True)[0]
        for b in S.buffers:
            b.fill_(fill)
        S.set_state(W.random_field_state(shape, Q, spread=0.2))
        S.step(5)
        out.append(S.get_state())
    assert torch.isfinite(out[0]).all()
    assert torch.equal(*out)


@pytest.mark.parametrize("Q", [27, 15])
@pytest.mark.parametrize("storage", ["f16", "bf16"])
@pytest.mark.parametrize("walls", [0, 3])
@pytest.mark.parametrize("form", [False, True])
@pytest.mark.parametrize("shape", [(3, 4, 9), (5, 6, 33)] + SHAPES)  # one- and two-cell
def test_16bit_step_matches_oracle(lbm, Q, storage, walls, form, shape):
    """One step from a state as stored against the FP64 oracle: what is stored is
    (f - w) / w, below 2 here, rounded up or down."""
    import oracle
    w = oracle.equilibrium(Q, np.ones((1, 1, 1)), np.zeros((3, 1, 1, 1)), np.zeros(3))
    S, om, F = _solver(lbm, Q, shape, walls, form, storage=storage)
    S.set_state(w * (1 + W.rng(15).uniform(-0.2, 0.2, (Q,) + shape)))
    f = S.get_state().cpu().numpy()
    S.step(1)
    want = oracle.run(Q, shape, f, F, om, 1, bc=walls)
    assert np.abs(want / w - 1).max() < 1.5  # and BF16 references below 0.5
    ulp = 2.0 ** (-10 if storage == "f16" else -7)
    assert (np.abs(S.get_state().cpu().numpy() - want) <= w * ulp + 2e-6).all()


@pytest.mark.parametrize("Q", [27, 15])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("walls", [0, 3])
@pytest.mark.parametrize("general", [False, True])
def test_adjoint_of_an_odd_row_equals_the_row_twice_over(lbm, Q, storage, walls, general):
    """The state is at rest in the 16-bit types (their rounding depends on the pair)."""
    shape = SHAPES[1]
    om = W.omegas(Q, 1 / 0.6)
    if general:
        om[9:] = 1.1
    f = W.random_field_state(shape, Q, spread=0.2 if storage == "f32" else 0.0)
    F = W.rng(16).uniform(-1e-2, 1e-2, (3,) + shape)
    lam = W.rng(17).standard_normal((Q,) + shape)
    got = []
    for k in (1, 2):
        S = lbm.Solver(Q, shape[:2] + (k * shape[2],), om, walls=walls, storage=storage,
                       force=np.concatenate([F] * k, -1))
        S.set_state(np.concatenate([f] * k, -1))
        a, b = S.new_adjoint_field(), S.new_adjoint_field()
        S.adjoint_view(a).copy_(torch.as_tensor(np.concatenate([lam] * k, -1)))
        gF = torch.zeros((3,) + S.shape, dtype=torch.float32, device="cuda")
        S.adjoint_step(S.current_buffer(), a, b, gF)
        got.append([v[..., :shape[2]].double().cpu().numpy() for v in (S.adjoint_view(b), gF)])
    for one, two in zip(*got):  # 1000 FP32 operations on O(1) values
        np.testing.assert_allclose(one, two, rtol=0, atol=1e-5 * np.abs(two).max())
