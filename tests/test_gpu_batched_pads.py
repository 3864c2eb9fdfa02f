"""Batches whose lattices lie on both sides of the FP32 ring's change of depth (needs a GB300).

The site-tensor ring of the FP32 sampler holds three tensors up to a bond pad of 32 and two
above, so a lattice of pad 32 may need more shared memory than one of the plan's largest pad.
Proposals and chains of such plans equal the single-lattice calls bit for bit, at the batch sizes
that choose 8 and 16 samples per warp, the narrower pad on the
wider rows and the other way round.
"""
import pytest

from paper_2104_13264_gb300 import instances

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SHIFT = 40


@pytest.mark.parametrize("n", [96, 4000])
@pytest.mark.parametrize("tile", [64, 128])
def test_mixed_pads_equal_single(n, tile):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_13264_gb300 import binding as B
    insts = [instances.random_small(Ly, Lx, 0.7, chi, seed=Lx + chi)
             for Ly, Lx, chi in ((7, 32, 36), (7, 32, 32), (7, 33, 29), (6, 15, 48), (5, 9, 3))]
    envs = B.build_envs_batched(insts, precisions=("f64", "f32"))
    assert [e.info()["pad"] for e in envs] == [36, 32, 32, 48, 4]
    for members in ([0, 1, 2], [3, 1, 4], [1, 0]):
        sub = [envs[i] for i in members]
        plan = B.Batch(sub, [n] * len(sub), chains=n // 2, precision="f32", tile=tile, order="cost")
        plan.set_step(11, 1)
        out = plan.sample(plan.alloc_proposals())
        chain = plan.init_chains(9)
        for i, e in enumerate(sub):
            ref = B.sample(e, n, seed=11, sample_offset=(i << SHIFT) + n, precision="f32")
            assert torch.equal(plan.view(out[0], i), ref[0])
            for a, b in zip(out[1:], ref[1:]):
                assert torch.equal(plan.rows(a, i), b)
            lq, E, _ = B.logq(e, plan.view(chain[0], i, chains=True), precision="f32")
            assert torch.equal(plan.rows(chain[1], i, chains=True), lq)
            assert torch.equal(plan.rows(chain[2], i, chains=True), E)
        plan.free()
    for e in envs:
        e.free()
