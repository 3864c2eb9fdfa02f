"""Wide rows, whose field factors, masks or bond dimensions do not sit in shared memory (needs a
GB300): BF16 proposals and the log q backward on both sides of each line.

The BF16 log q agrees with FP64 to 1e-4 relative (the precision's stated bound), the gradient
with the oracle's to 1e-3 per site (the bound of the gradient parity tests).  The gradient's
pad of 64 needs six rows.
"""
import numpy as np
import pytest

from oracle import tnmc
from paper_2104_13264_gb300 import instances

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("Lx", [203, 204, 509, 510, 3122, 3123, 3968])
def test_bf16_wide(Lx):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_13264_gb300 import binding as B
    env = B.Env.from_instance(instances.random_small(2, Lx, 0.7, 2, seed=Lx), precisions=("f64", "bf16"))
    sp, lq, E, fl = B.sample(env, 130, seed=5, precision="bf16")
    lq64, E64, fl64 = B.logq(env, sp, precision="f64")
    np.testing.assert_allclose(lq.cpu().numpy(), lq64.cpu().numpy(), rtol=1e-4)
    np.testing.assert_allclose(E.cpu().numpy(), E64.cpu().numpy(), rtol=1e-12)
    assert not fl.any() and not fl64.any()
    env.free()


def test_bf16_too_wide():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_13264_gb300 import binding as B
    env = B.Env.from_instance(instances.random_small(2, 3969, 0.7, 2, seed=1), precisions=("f64", "bf16"))
    with pytest.raises(B.TnmcError):
        B.sample(env, 4, seed=5, precision="bf16")
    env.free()


@pytest.mark.parametrize("Lx", [2630, 2631])
def test_grad_wide(Lx):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_13264_gb300 import binding as B
    inst = instances.random_small(6, Lx, 0.7, 64, seed=Lx)
    env = B.Env.from_instance(inst, precisions=("f64", "f32"))
    P = env.info()["pad"]
    assert P == 64
    ex = env.export()
    bd = ex["bond_dims"]
    ref = tnmc.Env(Lx, 6, inst.beta, 64, inst.Jh, inst.Jv, inst.h)
    ref.M = [[ex["tensors"][r, c, :bd[r, c], :, :bd[r, c + 1]].copy() for c in range(Lx)] for r in range(6)]
    sp = B.sample(env, 3, seed=7, precision="f32")[0].cpu().numpy()
    w = np.array([0.3, 1.0, 0.6])
    _, G = tnmc.logq_grad(ref, sp, w)
    grad = B.logq_backward(env, torch.from_numpy(sp).cuda(), torch.from_numpy(w).float().cuda())
    g = grad.cpu().numpy().reshape(6, Lx, P, 2, P)
    gmax = max(np.linalg.norm(G[r][c]) for r in range(6) for c in range(Lx))
    for r in range(6):
        for c in range(Lx):
            got = g[r, c, :G[r][c].shape[0], :, :G[r][c].shape[2]]
            assert np.linalg.norm(got - G[r][c]) <= 1e-3 * max(np.linalg.norm(G[r][c]), 1e-4 * gmax), (r, c)
    env.free()
