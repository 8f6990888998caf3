"""FP32 planes of more than 2^32 bytes, which take element offsets instead of byte
offsets.  A grid of three planes repeated along z evolves like the three alone; a
byte offset that wrapped would take a plane of another phase (the wrap, 1024
planes, is not a multiple of 3)."""
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


@pytest.mark.parametrize("Q,inplace", [(15, False), (15, True), (27, True)])
def test_repeated_planes_evolve_alike(lbm, Q, inplace):
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 200 << 30:
        pytest.skip("needs 200 GiB of free device memory")
    plane, times = (1024, 1024), 342  # 1026 x 2^20 elements
    g = torch.Generator(device="cuda").manual_seed(31)
    shape = (3,) + plane
    rho = torch.ones(shape, dtype=torch.float64, device="cuda")
    u = 0.1 * (torch.rand((3,) + shape, dtype=torch.float64, device="cuda", generator=g) - 0.5)
    fields = []
    for k in (1, times):
        S = lbm.Solver(Q, (3 * k,) + plane, W.omegas(Q, 1 / 0.6), force=(1e-4, 0, 0),
                       inplace=inplace)
        S.init_equilibrium(rho.repeat(k, 1, 1), u.repeat(1, k, 1, 1))
        torch.cuda.synchronize()
        S._keep = None
        S.step(3)
        fields.append(S.macroscopic())
        torch.cuda.synchronize()
        del S
        torch.cuda.empty_cache()
    # the instantiations differ in the code generator's fused operations: a few
    # roundings of values near 1 per step (2^-24 x 20 operations x 3 steps < 4e-6)
    (r1, u1), (r, v) = fields
    assert u1.std() > 1e-3
    assert (r.view((times,) + shape) - r1).abs().max() <= 4e-6
    for d in range(3):
        assert (v[d].view((times,) + shape) - u1[d]).abs().max() <= 4e-6
