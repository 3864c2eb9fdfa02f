"""Energies of real couplings (needs a GB300) against correctly rounded sums.

The couplings are held in 64-bit fixed point whose unit is 2^(e - 63) with e the exponent of the sum S
of their magnitudes (S < 2^e; one more where the roundings need it).  Each of the n terms is off by
at most half a unit, and the sum is rounded to FP64 once: |E - exact| <= n 2^(e - 63) + ulp(E).
A single large field must not cost the other couplings more than that.
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("field,beta", [(0.0, 0.5), (1e3, 0.05), (1e6, 1e-4)])
@pytest.mark.parametrize("Ly,Lx", [(48, 64), (5, 7), (1, 9), (6, 1)])
def test_energy_keeps_the_bits_of_small_couplings(Ly, Lx, field, beta):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_13264_gb300 import binding as B
    rng = np.random.default_rng(Ly * 100 + Lx)
    Jh, Jv = rng.standard_normal((Ly, Lx - 1)), rng.standard_normal((Ly - 1, Lx))
    h = 0.3 * rng.standard_normal((Ly, Lx))
    if field:
        h[Ly // 2, Lx // 3] = field
    env = B.Env(Jh, Jv, h, beta, 2, precisions=("f64", "f32", "bf16"))
    sp = rng.choice(np.array([-1, 1], dtype=np.int8), size=(9, Ly, Lx))
    n = Jh.size + Jv.size + h.size
    S = math.fsum(np.abs(np.concatenate([Jh.ravel(), Jv.ravel(), h.ravel()])))
    unit = 2.0 ** (math.frexp(S)[1] - 63)
    batch = B.Batch([env], [9], chains=1, precision="f64", tile=64)
    got = {p: B.logq(env, torch.from_numpy(sp).cuda(), precision=p)[1].cpu().numpy() for p in ("f64", "f32", "bf16")}
    got["batch"] = batch.logq(torch.from_numpy(sp).cuda().reshape(-1))[1].cpu().numpy()
    for k, s in enumerate(sp.astype(np.float64)):
        exact = -math.fsum(np.concatenate([(s[:, 1:] * s[:, :-1] * Jh).ravel(), (s[1:] * s[:-1] * Jv).ravel(),
                                           (s * h).ravel()]))
        for p, E in got.items():
            assert abs(E[k] - exact) <= n * unit + math.ulp(exact), (p, k)
    batch.free()
    env.free()
