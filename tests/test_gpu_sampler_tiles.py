"""Tile shapes of the FP64 and FP32 samplers (needs a GB300).

The launch picks the samples per warp from the batch size and the bond dimension.  A sample's
draw, log q and energy must not depend on that choice: the leading samples of batches of every
size class agree bit for bit, at bond dimensions on and off the tile edges, in both site
orders.  One batch per lattice is checked against the oracle on the same tensors (FP64 log q
to 1e-9, FP32 to 1e-4 relative, the precisions' stated bounds).
"""
import numpy as np
import pytest

from oracle import tnmc
from paper_2104_13264_gb300 import instances

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SIZES = (1, 37, 700, 1500, 3100, 9001, 15001, 33000, 41000)
# bond dimensions around the output blocks (4 lanes x 1, 2, 3, 4, 6, 8, 12, 16 bonds)
LATTICES = [(7, 9, 3), (6, 11, 5), (7, 13, 9), (8, 17, 13), (7, 15, 16), (7, 33, 17), (7, 19, 24), (8, 18, 32),
            (8, 16, 36), (9, 21, 50), (9, 20, 64), (3, 1, 2), (1, 6, 2), (5, 2, 4)]


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("Ly,Lx,chi", LATTICES)
def test_results_do_not_depend_on_the_tile(Ly, Lx, chi, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_13264_gb300 import binding as B
    inst = instances.random_small(Ly, Lx, 0.7, chi, seed=Ly * 100 + Lx)
    env = B.Env.from_instance(inst, precisions=("f64", "f32"))
    for order in ("raster", "snake"):
        env.set_order(order)
        big = B.sample(env, SIZES[-1], seed=5, sample_offset=9, precision=precision)
        for n in SIZES[:-1]:
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
        sp = big[0][:64].cpu().numpy()
        _, olq, oE, ofl = tnmc.logq(ref, sp)
        lq = big[1][:64].cpu().numpy()
        if precision == "f64":
            np.testing.assert_allclose(lq, olq, rtol=0, atol=1e-9)
        else:
            np.testing.assert_allclose(lq, olq, rtol=1e-4)
        np.testing.assert_allclose(big[2][:64].cpu().numpy(), oE, rtol=1e-12, atol=1e-12)
    env.free()
