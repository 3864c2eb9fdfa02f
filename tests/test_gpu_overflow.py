"""Environments whose weights overflow FP64 (needs a GB300).

The builders and samplers go on with truncated bonds, whatever the values are: the bond dimensions
are those of the formula, the status or the samples' flags report the overflow, every call returns,
and the next lattice's results are untouched.  Couplings with beta |J| of a few hundred make
infinities in the site products and NaN in their differences.
"""
import numpy as np
import pytest

from oracle import tnmc
from paper_2104_13264_gb300 import instances

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_13264_gb300 import binding
    binding.lib()
    return binding


def _good(B):
    inst = instances.random_small(6, 7, 0.8, 8, seed=2)
    env = B.Env.from_instance(inst)
    sp, lq, E, fl = B.sample(env, 40, seed=3)
    ref = tnmc.build_env(inst.Jh, inst.Jv, inst.h, inst.beta, inst.chi)
    osp, olq, oE, _ = tnmc.sample(ref, 40, seed=3)
    assert np.array_equal(sp.cpu().numpy(), osp) and np.abs(lq.cpu().numpy() - olq).max() < 1e-9
    env.free()


def _use(B, env, chi, gauge, reported):
    bd = env.export()["bond_dims"]
    for r in range(env.Ly):
        for c in range(env.Lx + 1):
            want = tnmc.bond_dim(chi, env.Lx, env.Ly, r, c)
            if gauge == "bond":       # the untruncated MPS of the row over the row below's bonds
                want = (1 if r == env.Ly - 1 else tnmc.bond_dim(chi, env.Lx, env.Ly, r + 1, c)) * (2 if 0 < c < env.Lx else 1)
            assert bd[r, c] == want, (r, c)
    for precision in ("f64", "f32", "bf16"):
        sp, lq, E, fl = B.sample(env, 70, seed=5, precision=precision)
        B.logq(env, sp, precision=precision)
        torch.cuda.synchronize()
        assert bool(((sp == 1) | (sp == -1)).all())
        reported |= env.status() != 0 or bool(fl.any())
    B.logq_backward(env, sp, torch.ones(70, device="cuda"))
    torch.cuda.synchronize()
    return reported


@pytest.mark.parametrize("beta", [150.0, 250.0, 400.0, 700.0])
@pytest.mark.parametrize("kind", ["pm", "field"])
@pytest.mark.parametrize("gauge,sweeps", [("spin", 0), ("bond", 0), ("spin", 1)])
def test_overflowing_environment_stays_in_bounds(B, beta, kind, gauge, sweeps):
    insts = [instances.ea_pm(6, 9, beta, 16, seed=3) if kind == "pm" else instances.random_small(7, 8, beta, 5, seed=3)]
    reported = False
    for inst in insts:
        env = B.Env.from_instance(inst, precisions=("f64", "f32", "bf16"), gauge=gauge, sweeps=sweeps)
        reported = _use(B, env, inst.chi, gauge, reported)
        env.free()
    assert reported or beta < 400.0
    _good(B)


def test_overflowing_batch_stays_in_bounds(B):
    insts = [instances.ea_pm(6, 9, 400.0, 16, seed=3), instances.random_small(6, 7, 0.8, 8, seed=2),
             instances.random_small(7, 8, 400.0, 5, seed=3)]
    envs = B.build_envs_batched(insts, precisions=("f64", "f32", "bf16"))
    single = B.Env.from_instance(insts[1], precisions=("f64", "f32"))
    assert np.array_equal(envs[1].export()["tensors"], single.export()["tensors"])
    for e, inst in zip(envs, insts):
        _use(B, e, inst.chi, "spin", False)
    for e in (*envs, single):
        e.free()


@pytest.mark.parametrize("form", ["thread", "shared", "warp"])
@pytest.mark.parametrize("gauge", ["spin", "bond"])
@pytest.mark.parametrize("beta", [60.0, 400.0])
def test_overflowing_cube_stays_in_bounds(B, monkeypatch, form, gauge, beta):
    monkeypatch.setenv("TNMC_3D_KERNEL", form)
    env = B.Env3D.from_instance(instances.cubic_random(3, 4, 3, beta, 2, 2, seed=3), gauge=gauge)
    for precision in ("f64", "f32"):
        sp, lq, E, fl = B.sample3d(env, 70, seed=5, precision=precision)
        B.logq3d(env, sp, precision=precision)
        torch.cuda.synchronize()
        assert bool(((sp == 1) | (sp == -1)).all())
    env.free()
    monkeypatch.delenv("TNMC_3D_KERNEL")
    _good(B)
