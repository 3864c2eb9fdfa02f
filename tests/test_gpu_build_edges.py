"""Edges of the FP64 builder (needs a GB300): row pairs on both sides of every lane split of the
Jacobi rounds, and column counts that leave every remainder in the packed reductions of the QR,
with and without fields (parity sectors), against the oracle's builder.

Bounds as in the builder's parity tests: 1e-9 for log Z, scales and singular values, 1e-10 for
the orthonormality of the sites.
"""
import numpy as np
import pytest

from oracle import tnmc
from paper_2104_13264_gb300 import instances

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("Ly,Lx,chi", [(2, 2, 2), (3, 5, 3), (4, 7, 5), (5, 9, 7), (5, 9, 8), (5, 10, 9), (6, 11, 16),
                                       (6, 11, 17), (7, 13, 31), (7, 13, 33), (8, 14, 64)])
@pytest.mark.parametrize("field", [False, True])
def test_build_edges(Ly, Lx, chi, field):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_13264_gb300 import binding as B
    inst = instances.random_small(Ly, Lx, 0.7, chi, seed=chi, hscale=0.3 if field else 0.0)
    ref = tnmc.build_env(inst.Jh, inst.Jv, inst.h, inst.beta, inst.chi)
    env = B.Env.from_instance(inst, precisions=("f64",))
    assert env.status() == 0
    ex = env.export()
    assert ex["logZ"] == pytest.approx(ref.logZ, abs=1e-9 * max(1.0, abs(ref.logZ)))
    np.testing.assert_allclose(ex["log_scale"], ref.log_scale, rtol=1e-9, atol=1e-9)
    for (r, c), s in ref.sv.items():
        np.testing.assert_allclose(ex["sv"][r, c, :s.size], s, atol=1e-9)
    for r in range(Ly):
        for c in range(1, Lx):
            a, b = ex["bond_dims"][r, c], ex["bond_dims"][r, c + 1]
            A = ex["tensors"][r, c, :a, :, :b].reshape(a, -1)
            nz = np.linalg.norm(A, axis=1) > 0.5
            np.testing.assert_allclose(A[nz] @ A[nz].T, np.eye(int(nz.sum())), atol=1e-10)
            assert np.all(np.linalg.norm(A[~nz], axis=1) == 0)
    env.free()
