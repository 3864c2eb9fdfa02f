"""The 3D sampler's working matrices in shared memory, FP64 at bonds that fit (needs a GB300).

A CTA is one warp; a sample's slice holds D K^2 + K^2 + K + 2 D K^2 values, K = D chi (D: the bond the
sampler sees, doubled in the bond basis).  The form is taken only where 32 slices of 8 bytes fit the
232448 bytes a CTA may have, so the shapes here are checked against that first: at (3, 4) the forced
form would silently be the scratch form, and comparing it shows nothing.
"""
import pytest

from paper_2104_13264_gb300 import instances

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _slice_bytes(D, chi):
    K = D * chi
    return (K * K * D + K * K + K + 2 * K * D * K) * 32 * 8


@pytest.mark.parametrize("shape,D,chi,gauge", [((2, 6, 1), 2, 4, "spin"), ((3, 4, 3), 4, 2, "spin"),
                                               ((3, 3, 4), 2, 2, "bond"), ((2, 1, 5), 1, 7, "spin")])
def test_shared_form_equals_scratch_form_f64(monkeypatch, shape, D, chi, gauge):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_13264_gb300 import binding as B
    assert _slice_bytes(2 * D if gauge == "bond" else D, chi) <= 232448 < _slice_bytes(3, 4)
    env = B.Env3D.from_instance(instances.cubic_random(*shape, 0.6, D, chi, seed=3), gauge=gauge)
    out = {}
    for form in ("thread", "shared"):
        monkeypatch.setenv("TNMC_3D_KERNEL", form)
        out[form] = B.sample3d(env, 77, seed=5)
        lq, E, fl = B.logq3d(env, out[form][0])
        assert torch.equal(lq, out[form][1]) and torch.equal(E, out[form][2])
    for a, b in zip(out["thread"], out["shared"]):
        assert torch.equal(a, b)
    env.free()
