"""Tile edges of the log q backward (needs a GB300).

Bond dimensions and batch sizes on and off the kernel's 32-sample tile and output blocks, and
a gradient buffer that is only 4-byte aligned, against the oracle's gradient on the same
seeded tensors: 1e-3 relative per site (the bound of the gradient parity tests).
"""
import ctypes

import numpy as np
import pytest

from oracle import tnmc
from paper_2104_13264_gb300 import instances

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("Ly,Lx,chi,B,shift", [(4, 1, 2, 33, 0), (1, 6, 2, 1, 0), (4, 9, 5, 31, 1), (6, 13, 17, 32, 0),
                                               (6, 13, 24, 70, 2), (7, 14, 36, 33, 0), (7, 13, 50, 64, 1)])
def test_grad_tile_edges(Ly, Lx, chi, B, shift):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_13264_gb300 import binding
    inst = instances.random_small(Ly, Lx, 0.7, chi, seed=chi)
    shapes = [(tnmc.bond_dim(chi, Lx, Ly, r, c), 2, tnmc.bond_dim(chi, Lx, Ly, r, c + 1))
              for r in range(Ly) for c in range(Lx)]
    ts = instances.random_tensors(shapes, seed=chi)
    ref = tnmc.Env(Lx, Ly, inst.beta, chi, inst.Jh, inst.Jv, inst.h)
    ref.M = [[ts[r * Lx + c] for c in range(Lx)] for r in range(Ly)]
    env = binding.Env.from_instance(inst, precisions=("f64", "f32"))
    P = env.info()["pad"]
    flat = np.zeros((Ly, Lx, P, 2, P), dtype=np.float32)
    for r in range(Ly):
        for c in range(Lx):
            t = ts[r * Lx + c]
            flat[r, c, :t.shape[0], :, :t.shape[2]] = t
    binding.set_params(env, torch.from_numpy(flat.reshape(-1)).cuda())
    sp, _, _, _ = tnmc.sample(ref, B, seed=7)
    w = np.random.default_rng(chi).random(B)
    _, G = tnmc.logq_grad(ref, sp, w)
    spins, wt = torch.from_numpy(sp).cuda(), torch.from_numpy(w).float().cuda()
    buf = torch.full((flat.size + 4,), 7.0, dtype=torch.float32, device="cuda")
    st = binding.lib().tnmc_logq_backward(env.handle, B, ctypes.c_void_p(spins.data_ptr()),
                                          ctypes.c_void_p(wt.data_ptr()), ctypes.c_void_p(buf.data_ptr() + 4 * shift),
                                          ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0
    out = buf.cpu().numpy()
    assert np.all(out[:shift] == 7.0) and np.all(out[shift + flat.size:] == 7.0)
    g = out[shift:shift + flat.size].reshape(flat.shape)
    gmax = max(np.linalg.norm(G[r][c]) for r in range(Ly) for c in range(Lx))
    for r in range(Ly):
        for c in range(Lx):
            got = g[r, c, :G[r][c].shape[0], :, :G[r][c].shape[2]]
            assert np.linalg.norm(got - G[r][c]) <= 1e-3 * max(np.linalg.norm(G[r][c]), 1e-4 * gmax), (r, c)
            rest = g[r, c].copy()
            rest[:G[r][c].shape[0], :, :G[r][c].shape[2]] = 0.0
            assert not rest.any()
    env.free()
