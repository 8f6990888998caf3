"""Rows of odd length: the last thread of a row has one cell.  A periodic row
of n cells and the same row twice over (2n cells, even) evolve alike, so the
two are compared cell by cell: equal FP32 arithmetic up to the code generator's
choice of fused operations, a few roundings of values below 1 per step
(2^-24 x 20 operations x 3 steps < 4e-6)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROWS = [1, 3, 5, 31, 33, 255, 257]


@pytest.fixture(scope="module")
def lbm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1202_6081_gb300 import build
    from paper_1202_6081_gb300 import lbm as mod
    build()
    mod.load()
    return mod


def _rates(Q, general):
    om = W.omegas(Q, 1 / 0.6)
    if general:
        om[9:] = 1.1
    return om


@pytest.mark.parametrize("Q", [27, 15])
@pytest.mark.parametrize("walls", [0, 3])
@pytest.mark.parametrize("general", [False, True])
@pytest.mark.parametrize("n", ROWS)
def test_odd_row_equals_the_row_twice_over(lbm, Q, walls, general, n):
    shape = (3, 4, n)
    f = W.random_field_state(shape, Q, spread=0.2)
    F = W.rng(3).uniform(-1e-2, 1e-2, (3,) + shape)
    lam = W.rng(4).standard_normal((Q,) + shape)
    got = []
    for k in (1, 2):
        S = lbm.Solver(Q, shape[:2] + (k * n,), _rates(Q, general), walls=walls,
                       force=np.concatenate([F] * k, -1))
        S.set_state(np.concatenate([f] * k, -1))
        a, b = S.new_adjoint_field(), S.new_adjoint_field()
        S.adjoint_view(a).copy_(torch.as_tensor(np.concatenate([lam] * k, -1)))
        gF = torch.zeros((3,) + S.shape, dtype=torch.float32, device="cuda")
        S.adjoint_step(S.current_buffer(), a, b, gF)
        S.step(3)
        got.append([v[..., :n].double().cpu().numpy()
                    for v in (S.get_state(), S.adjoint_view(b), gF)])
    np.testing.assert_allclose(got[0][0], got[1][0], rtol=0, atol=4e-6)
    for one, two in zip(got[0][1:], got[1][1:]):  # 1000 FP32 operations on O(1) values
        np.testing.assert_allclose(one, two, rtol=0, atol=1e-5 * np.abs(two).max())


@pytest.mark.parametrize("Q", [27, 15])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("n", ROWS)
def test_results_do_not_depend_on_the_padding(lbm, Q, storage, n):
    shape = (3, 4, n)
    out = []
    for fill in (0x00, 0xff):  # zeros, NaNs
        S = lbm.Solver(Q, shape, _rates(Q, False), walls=2, force=(1e-4, 0, 0), storage=storage)
        for b in S.buffers:
            b.fill_(fill)
        S.set_state(W.random_field_state(shape, Q, spread=0.2))
        S.step(5)
        out.append(S.get_state().cpu().numpy())
    assert np.isfinite(out[0]).all()
    np.testing.assert_array_equal(out[0], out[1])


@pytest.mark.parametrize("Q", [27, 15])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("walls", [0, 3])
@pytest.mark.parametrize("n", [2, 30, 34, 72, 130, 258, 384])
def test_ragged_rows_in_place_equal_two_buffers_bitwise(lbm, Q, storage, walls, n):
    shape = (4, 5, n)
    states = []
    for inplace in (False, True):
        S = lbm.Solver(Q, shape, _rates(Q, False), walls=walls, force=(1e-4, -1e-4, 0),
                       storage=storage, inplace=inplace)
        S.set_state(W.random_field_state(shape, Q, spread=0.2))
        S.step(5)
        states.append(S.get_state())
    assert torch.equal(*states)
