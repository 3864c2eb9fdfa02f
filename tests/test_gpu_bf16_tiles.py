"""Edges of the BF16 tensor-core sampler (needs a GB300): bond dimensions on both sides of every
K step of 16, odd widths (a Philox pair that spans two rows), one-site rows, non-integer
couplings, and batches below, at and above a 128-sample tile and one wave of CTAs.

A sample's results do not depend on the batch size, forced evaluation reproduces them bit for
bit, and log q matches the oracle on the environment rounded to the same hi + lo pairs to 1e-4
relative (the precision's stated bound); energies are exact to rounding.
"""
import numpy as np
import pytest

from oracle import tnmc
from paper_2104_13264_gb300 import instances

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("Ly,Lx,chi", [(5, 1, 2), (1, 7, 2), (5, 9, 6), (6, 11, 16), (6, 13, 17), (7, 15, 32),
                                       (7, 13, 33), (8, 15, 48), (8, 15, 49), (8, 14, 64)])
def test_bf16_edges(Ly, Lx, chi):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_13264_gb300 import binding as B
    inst = instances.random_small(Ly, Lx, 0.7, chi, seed=Ly * 100 + Lx)
    env = B.Env.from_instance(inst, precisions=("f64", "bf16"))
    big = B.sample(env, 40001, seed=5, sample_offset=9, precision="bf16")
    for n in (1, 31, 128, 129, 5000):
        got = B.sample(env, n, seed=5, sample_offset=9, precision="bf16")
        for a, b in zip(got, big):
            assert torch.equal(a, b[:n]), n
        lq, E, fl = B.logq(env, got[0], precision="bf16")
        assert torch.equal(lq, got[1]) and torch.equal(E, got[2]) and torch.equal(fl, got[3])
    ex = env.export()
    ref = tnmc.Env(Lx, Ly, inst.beta, chi, inst.Jh, inst.Jv, inst.h)
    bd = ex["bond_dims"]
    ref.M = [[ex["tensors"][r, c, :bd[r, c], :, :bd[r, c + 1]].copy() for c in range(Lx)] for r in range(Ly)]
    sp = big[0][:64].cpu().numpy()
    _, olq, oE, _ = tnmc.logq(tnmc.env_bf16(ref), sp)
    np.testing.assert_allclose(big[1][:64].cpu().numpy(), olq, rtol=1e-4)
    np.testing.assert_allclose(big[2][:64].cpu().numpy(), oE, rtol=1e-12, atol=1e-12)
    env.free()
