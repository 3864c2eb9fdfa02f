"""The log q backward of small bonds and large batches (needs a GB300).

One thread per sample from 64 samples per SM on at a pad of 4, from 256 on at a pad of 8.  Both sides of
the lines (152 SMs), both tile sizes, several tiles per CTA, partly filled tiles, rows and columns of
one site and samples without weight, against the oracle's gradient on the same tensors: 1e-3
relative per site (the bound of the gradient parity tests).
"""
import numpy as np
import pytest

from oracle import tnmc
from paper_2104_13264_gb300 import instances

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("Ly,Lx,chi,n", [(4, 9, 3, 9727), (4, 9, 3, 9728), (6, 13, 4, 20001), (6, 13, 4, 39001),
                                         (1, 6, 2, 9999), (4, 1, 2, 9999), (5, 8, 7, 38911), (5, 8, 7, 38913),
                                         (2, 6, 2, 400001)])
def test_small_bonds_large_batches(Ly, Lx, chi, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_13264_gb300 import binding as B
    inst = instances.random_small(Ly, Lx, 0.7, chi, seed=chi)
    env = B.Env.from_instance(inst, precisions=("f64", "f32"))
    P = env.info()["pad"]
    assert P == (4 if chi <= 4 else 8)
    ex = env.export()
    bd = ex["bond_dims"]
    ref = tnmc.Env(Lx, Ly, inst.beta, chi, inst.Jh, inst.Jv, inst.h)
    ref.M = [[ex["tensors"][r, c, :bd[r, c], :, :bd[r, c + 1]].astype(np.float32).astype(np.float64)
              for c in range(Lx)] for r in range(Ly)]
    sp = B.sample(env, n, seed=7)[0]
    w = np.random.default_rng(chi).random(n)
    w[::7] = 0.0
    _, G = tnmc.logq_grad(ref, sp.cpu().numpy(), w)
    g = B.logq_backward(env, sp, torch.from_numpy(w).float().cuda()).cpu().numpy().reshape(Ly, Lx, P, 2, P)
    gmax = max(np.linalg.norm(G[r][c]) for r in range(Ly) for c in range(Lx))
    for r in range(Ly):
        for c in range(Lx):
            got = g[r, c, :G[r][c].shape[0], :, :G[r][c].shape[2]]
            assert np.linalg.norm(got - G[r][c]) <= 1e-3 * max(np.linalg.norm(G[r][c]), 1e-4 * gmax), (r, c)
            rest = g[r, c].copy()
            rest[:G[r][c].shape[0], :, :G[r][c].shape[2]] = 0.0
            assert not rest.any()
    env.free()
