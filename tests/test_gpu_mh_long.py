"""Long MH scans of few chains (needs a GB300): the form with one CTA per chain links accepted
proposals in parallel, so it must reproduce the oracle's sequential scan at every acceptance
rate, across its blocks of proposals, from starts outside q's support, past proposals that can
never be accepted, and where a decision is left to the FP64 rule.
"""
import numpy as np
import pytest

from oracle import philox, tnmc
from paper_2104_13264_gb300 import instances

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("C,T,spread,start", [(1, 10000, 0.1, False), (2, 4097, 3.0, True), (3, 2500, 30.0, False),
                                              (5, 128, 1.0, True), (1, 12289, 8.0, True), (40, 333, 2.0, False)])
def test_long_scan_matches_the_oracle(C, T, spread, start):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_13264_gb300 import binding as B
    inst = instances.ferromagnet(2, 3, 0.5, 2)
    env = B.Env.from_instance(inst)
    rng = np.random.default_rng(C * 100003 + T)
    seed, off = 17, 5
    lq = spread * rng.standard_normal(C * T)
    E = rng.integers(-7, 8, size=C * T).astype(np.float64)
    lq[rng.random(C * T) < 0.02] = -np.inf
    lq[rng.random(C * T) < 0.01] = np.nan
    clq = np.full(C, -np.inf if start else 0.0)
    cE = np.zeros(C)
    # a few decisions inside their band: Delta within 1e-12 of log u of the state they meet
    for i in range(C):
        a, have = -inst.beta * cE[i] - clq[i], not start
        u = philox.mh_uniform(seed, np.uint64(off) + np.arange(T, dtype=np.uint64), np.uint64(i))
        for j in range(T):
            t = i * T + j
            if have and rng.random() < 0.03 and u[j] > 0:
                lq[t] = -inst.beta * E[t] - (a + np.log(u[j]) + rng.choice([-3e-13, 2e-13, 5e-13]))
            if np.isfinite(lq[t]):
                at = -inst.beta * E[t] - lq[t]
                if not have or u[j] < np.exp(min(0.0, at - a)):
                    a, have = at, True
    sp = np.where(rng.random((C * T, inst.Ly, inst.Lx)) < 0.5, 1, -1).astype(np.int8)
    csp = -np.ones((C, inst.Ly, inst.Lx), dtype=np.int8)
    want, wsp, wlq, wE = tnmc.mh_scan(inst.beta, C, T, sp, lq, E, csp.copy(), clq.copy(), cE.copy(), seed=seed,
                                      step_offset=off)
    dev = [torch.from_numpy(x.copy()).cuda() for x in (sp, lq, E, csp, clq, cE)]
    count = torch.zeros(1, dtype=torch.int64, device="cuda")
    acc = B.mh_step(env, C, T, tuple(dev[:3]), tuple(dev[3:]), seed=seed, step_offset=off, n_accepted=count)
    acc = acc.cpu().numpy().astype(bool)
    assert np.array_equal(acc, want), np.nonzero(acc != want)[0][:10]
    assert int(count) == int(want.sum()) and want.any() and (~want).any()
    assert np.array_equal(dev[3].cpu().numpy(), wsp)
    assert np.array_equal(dev[4].cpu().numpy(), wlq) and np.array_equal(dev[5].cpu().numpy(), wE)
    env.free()
