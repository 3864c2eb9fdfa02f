"""Wide rows in the FP64 and FP32 samplers (needs a GB300).

From a few hundred (FP64) or about a thousand columns (FP32) on, the launch keeps field factors and
bond dimensions in global memory and picks other tile shapes.  A sample must not depend on the
choice: the leading samples of batches of every size class agree bit for bit in both site orders,
with the batched form and the call without allocations, and with the oracle on the same tensors
(FP64 log q to 1e-9 absolute per thousand sites, FP32 to 1e-4 relative, the precisions' bounds).
"""
import ctypes

import numpy as np
import pytest

from oracle import tnmc
from paper_2104_13264_gb300 import instances

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _noalloc(B, env, precision, n, seed, offset):
    dev = torch.device("cuda")
    out = (torch.empty((n, env.Ly, env.Lx), dtype=torch.int8, device=dev), torch.empty(n, dtype=torch.float64, device=dev),
           torch.empty(n, dtype=torch.float64, device=dev), torch.empty(n, dtype=torch.int32, device=dev))
    st = B.lib().tnmc_sample_noalloc(env.handle, B.PRECISIONS[precision], n, seed, offset,
                                     *(ctypes.c_void_p(t.data_ptr()) for t in out),
                                     ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0, B.lib().tnmc_last_error()
    return out


def _check(precision, Ly, Lx, chi, sizes):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_13264_gb300 import binding as B
    inst = instances.random_small(Ly, Lx, 0.7, chi, seed=Lx)
    env = B.Env.from_instance(inst, precisions=("f64", "f32"))
    for order in ("raster", "snake"):
        env.set_order(order)
        big = B.sample(env, sizes[-1], seed=5, sample_offset=9, precision=precision)
        for n in sizes[:-1]:
            got = B.sample(env, n, seed=5, sample_offset=9, precision=precision)
            for a, b in zip(got, big):
                assert torch.equal(a, b[:n]), (order, n)
            lq, E, fl = B.logq(env, got[0], precision=precision)
            assert torch.equal(lq, got[1]) and torch.equal(E, got[2]) and torch.equal(fl, got[3])
        ex = env.export()
        ref = tnmc.Env(Lx, Ly, inst.beta, chi, inst.Jh, inst.Jv, inst.h)
        bd = ex["bond_dims"]
        ref.M = [[ex["tensors"][r, c, :bd[r, c], :, :bd[r, c + 1]].copy() for c in range(Lx)] for r in range(Ly)]
        ref.order = order
        _, olq, oE, _ = tnmc.logq(ref, big[0][:4].cpu().numpy())
        lq = big[1][:4].cpu().numpy()
        if precision == "f64":
            np.testing.assert_allclose(lq, olq, rtol=0, atol=1e-12 * Lx * Ly)
        else:
            np.testing.assert_allclose(lq, olq, rtol=1e-4)
        np.testing.assert_allclose(big[2][:4].cpu().numpy(), oE, rtol=1e-12, atol=1e-11)
    n = sizes[1]
    plan = B.Batch([env, env], [n, n], chains=1, precision=precision)
    plan.set_step(5, 1)
    out = plan.sample(plan.alloc_proposals())
    one = B.sample(env, n, seed=5, sample_offset=n, precision=precision)
    for a, b in zip(out[1:], one[1:]):
        assert torch.equal(plan.rows(a, 0), b)
    for a, b in zip(_noalloc(B, env, precision, n, 5, n), one):
        assert torch.equal(a, b)
    plan.free()
    env.free()


@pytest.mark.parametrize("Ly,Lx,chi,sizes", [(2, 480, 2, (3, 1500, 9001, 41000)), (4, 700, 5, (5, 1500, 15001, 33000)),
                                             (2, 4096, 2, (1, 700, 9001, 33000)), (6, 1100, 20, (2, 1500, 4001))])
def test_f64_wide(Ly, Lx, chi, sizes):
    _check("f64", Ly, Lx, chi, sizes)


@pytest.mark.parametrize("Ly,Lx,chi,sizes", [(2, 1300, 2, (3, 1500, 9001, 41000)), (4, 2048, 5, (5, 4000, 15001, 33000)),
                                             (2, 4096, 2, (1, 1500, 9001, 66000)), (5, 3000, 13, (2, 1500, 4001, 41000)),
                                             (6, 2100, 20, (2, 1500, 9001)), (7, 1200, 50, (2, 3100, 9001))])
def test_f32_wide(Ly, Lx, chi, sizes):
    _check("f32", Ly, Lx, chi, sizes)
