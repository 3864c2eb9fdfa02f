"""Blocks of the MH scan with one CTA per chain (needs a GB300).

The block of proposals is the largest that leaves all chains' CTAs resident, down to 512, so the
number of chains decides how many blocks a scan has.  Decisions, chain states and counts equal the
oracle's sequential scan at every block size, with proposals that can never be accepted, and
across blocks without an acceptance (the spread of 200 accepts a few proposals of thousands).
"""
import numpy as np
import pytest

from oracle import tnmc
from paper_2104_13264_gb300 import instances

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("C,T", [(150, 4500), (300, 4200), (300, 2049), (700, 1600), (700, 1024), (1100, 1055),
                                 (2048, 600), (1100, 512)])
@pytest.mark.parametrize("spread", [0.5, 200.0])
def test_blocks_match_the_oracle(C, T, spread):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_13264_gb300 import binding as B
    inst = instances.ferromagnet(2, 3, 0.5, 2)
    env = B.Env.from_instance(inst)
    rng = np.random.default_rng(C + T)
    lq = spread * rng.standard_normal(C * T)
    E = rng.integers(-7, 8, size=C * T).astype(np.float64)
    lq[rng.random(C * T) < 0.02] = -np.inf
    clq, cE = np.zeros(C), np.zeros(C)
    clq[::3] = -np.inf      # starts outside q's support
    sp = np.where(rng.random((C * T, inst.Ly, inst.Lx)) < 0.5, 1, -1).astype(np.int8)
    csp = -np.ones((C, inst.Ly, inst.Lx), dtype=np.int8)
    want, wsp, wlq, wE = tnmc.mh_scan(inst.beta, C, T, sp, lq, E, csp.copy(), clq.copy(), cE.copy(), seed=9,
                                      step_offset=4)
    dev = [torch.from_numpy(x.copy()).cuda() for x in (sp, lq, E, csp, clq, cE)]
    count = torch.zeros(1, dtype=torch.int64, device="cuda")
    acc = B.mh_step(env, C, T, tuple(dev[:3]), tuple(dev[3:]), seed=9, step_offset=4, n_accepted=count)
    assert np.array_equal(acc.cpu().numpy().astype(bool), want)
    assert int(count) == int(want.sum())
    assert np.array_equal(dev[3].cpu().numpy(), wsp)
    assert np.array_equal(dev[4].cpu().numpy(), wlq) and np.array_equal(dev[5].cpu().numpy(), wE)
    env.free()
