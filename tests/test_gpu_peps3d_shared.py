"""The 3D sampler's working matrices in shared memory (needs a GB300): the same operations in the
same order as from global scratch, so spins, log q, energies and flags agree bit for bit, in both
precisions, at a partly filled warp, and on boxes that are one site wide."""
import pytest

from paper_2104_13264_gb300 import instances

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("shape,D,chi,gauge", [((3, 4, 5), 2, 2, "bond"), ((3, 4, 5), 2, 2, "spin"),
                                               ((2, 1, 6), 2, 3, "spin"), ((2, 6, 1), 3, 4, "spin"),
                                               ((2, 3, 3), 1, 1, "bond")])
@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_shared_form_equals_scratch_form(monkeypatch, shape, D, chi, gauge, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_13264_gb300 import binding as B
    env = B.Env3D.from_instance(instances.cubic_random(*shape, 0.6, D, chi, seed=3), gauge=gauge)
    out = {}
    for form in ("thread", "shared"):
        monkeypatch.setenv("TNMC_3D_KERNEL", form)
        out[form] = B.sample3d(env, 77, seed=5, precision=precision)
        lq, E, fl = B.logq3d(env, out[form][0], precision=precision)
        assert torch.equal(lq, out[form][1]) and torch.equal(E, out[form][2])
    for a, b in zip(out["thread"], out["shared"]):
        assert torch.equal(a, b)
    env.free()
