"""Strong vertical bonds (needs a GB300): beta |Jv| up to the end of FP32's range.

A row's field factors are exp(+-beta Jv).  The FP32 sampler stays unflagged as long as a single
factor fits FP32 (beta |Jv| < 88), and its log q agrees with FP64 to 1e-4 relative (the precision's
stated bound), whatever the signs of neighbouring bonds are; a batch equals the single calls.  The
BF16 sampler, whose accumulator holds two factors, does the same up to 44.  The gradient agrees with
the oracle's on the same tensors to 1e-3 per site (the bound of the gradient parity tests).
"""
import numpy as np
import pytest

from oracle import tnmc

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _lattice(Ly, Lx, beta, seed):
    """Vertical bonds of magnitude 0.9 to 1, everything else of order 1 / beta."""
    r = np.random.default_rng(seed)
    Jh = 0.7 / beta * r.standard_normal((Ly, Lx - 1))
    Jv = r.choice([-1.0, 1.0], size=(Ly - 1, Lx)) * r.uniform(0.9, 1.0, size=(Ly - 1, Lx))
    h = 0.3 / beta * r.standard_normal((Ly, Lx))
    return Jh, Jv, h


@pytest.mark.parametrize("beta", [19.0, 21.0, 30.0, 48.0, 84.0])
@pytest.mark.parametrize("Ly,Lx,chi", [(6, 9, 4), (7, 13, 20), (7, 14, 40)])
def test_f32_strong_bonds(Ly, Lx, chi, beta):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_13264_gb300 import binding as B
    env = B.Env(*_lattice(Ly, Lx, beta, chi), beta, chi, precisions=("f64", "f32"))
    for n in (300, 20000):
        for order in ("raster", "snake"):
            env.set_order(order)
            sp, lq, E, fl = B.sample(env, n, seed=5, precision="f32")
            lq64, _, fl64 = B.logq(env, sp, precision="f64")
            assert not fl.any() and not fl64.any()
            np.testing.assert_allclose(lq.cpu().numpy(), lq64.cpu().numpy(), rtol=1e-4)
        plan = B.Batch([env, env], [n, n], chains=n // 2, precision="f32")
        plan.set_step(5, 0)
        out = plan.sample(plan.alloc_proposals())
        assert torch.equal(plan.view(out[0], 0), sp) and torch.equal(plan.rows(out[1], 0), lq)
        plan.free()
    env.free()


def test_f32_batch_of_strong_and_weak_bonds():
    """One strong lattice takes the whole plan to the other form, which leaves the weak ones' bits."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_13264_gb300 import binding as B
    envs = [B.Env(*_lattice(6, 9, 48.0, 1), 48.0, 4, precisions=("f64", "f32")),
            B.Env(*_lattice(7, 13, 2.0, 2), 2.0, 20, precisions=("f64", "f32"))]
    for n in (60, 30000):
        plan = B.Batch(envs, [n, n], chains=n // 2, precision="f32")
        plan.set_step(5, 1)
        out = plan.sample(plan.alloc_proposals())
        for i, e in enumerate(envs):
            ref = B.sample(e, n, seed=5, sample_offset=(i << 40) + n, precision="f32")
            assert torch.equal(plan.view(out[0], i), ref[0])
            for a, b in zip(out[1:], ref[1:]):
                assert torch.equal(plan.rows(a, i), b)
        plan.free()
    for e in envs:
        e.free()


@pytest.mark.parametrize("beta", [19.0, 21.0, 32.0, 42.0])
@pytest.mark.parametrize("Ly,Lx,chi", [(6, 9, 4), (7, 13, 20), (7, 14, 40)])
def test_bf16_strong_bonds(Ly, Lx, chi, beta):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_13264_gb300 import binding as B
    env = B.Env(*_lattice(Ly, Lx, beta, chi), beta, chi, precisions=("f64", "bf16"))
    sp, lq, E, fl = B.sample(env, 300, seed=5, precision="bf16")
    lq64, _, fl64 = B.logq(env, sp, precision="f64")
    assert not fl.any() and not fl64.any()
    np.testing.assert_allclose(lq.cpu().numpy(), lq64.cpu().numpy(), rtol=1e-4)
    env.free()


@pytest.mark.parametrize("beta", [19.0, 21.0, 32.0, 42.0])
@pytest.mark.parametrize("Ly,Lx,chi,n", [(6, 9, 4, 40), (7, 13, 20, 40), (7, 14, 40, 40), (6, 9, 4, 10000)])
def test_grad_strong_bonds(Ly, Lx, chi, n, beta):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_13264_gb300 import binding as B
    Jh, Jv, h = _lattice(Ly, Lx, beta, chi)
    env = B.Env(Jh, Jv, h, beta, chi, precisions=("f64", "f32"))
    P = env.info()["pad"]
    ex = env.export()
    bd = ex["bond_dims"]
    ref = tnmc.Env(Lx, Ly, beta, chi, Jh, Jv, h)
    ref.M = [[ex["tensors"][r, c, :bd[r, c], :, :bd[r, c + 1]].astype(np.float32).astype(np.float64)
              for c in range(Lx)] for r in range(Ly)]
    sp = B.sample(env, n, seed=7)[0].cpu().numpy()
    w = np.random.default_rng(chi).random(n)
    _, G = tnmc.logq_grad(ref, sp, w)
    grad = B.logq_backward(env, torch.from_numpy(sp).cuda(), torch.from_numpy(w).float().cuda())
    g = grad.cpu().numpy().reshape(Ly, Lx, P, 2, P)
    gmax = max(np.linalg.norm(G[r][c]) for r in range(Ly) for c in range(Lx))
    for r in range(Ly):
        for c in range(Lx):
            got = g[r, c, :G[r][c].shape[0], :, :G[r][c].shape[2]]
            assert np.linalg.norm(got - G[r][c]) <= 1e-3 * max(np.linalg.norm(G[r][c]), 1e-4 * gmax), (r, c)
    env.free()
