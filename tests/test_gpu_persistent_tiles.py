"""Collide-stream tiles of the persistent batched form with 16-bit storage: a
cell per thread where the tile has at most half as many blocks as the CTA has
warps, else two (a packed pair)."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

STEPS = 2


@pytest.mark.parametrize("q", [19, 27])
@pytest.mark.parametrize("storage,u", [("f16", 2.0 ** -11), ("bf16", 2.0 ** -8)])
def test_16bit_tiles(q, storage, u):
    """Against FP32 storage: every store rounds f - w_p by u at most, and a value
    goes through the import and, per substep of the finest of the three levels
    (4 a coarse step), a collision and an exchange."""
    from oracle.lattice import VelocitySet
    from paper_2308_08085_gb300 import AmrBatch, AmrLBM, build as b
    b.build()
    w = VelocitySet(3, q).w
    cfgs = [W.cavity(dim=3, q=q, n=12, ny=8, nz=8, re=50.0, max_levels=3, max_blocks=480),
            W.cavity(dim=3, q=q, n=8, re=50.0, max_levels=1, max_blocks=8)]

    def forest(i, storage):
        sim = AmrLBM(cfgs[i], storage=storage)
        for seed in (3, 4):
            m = W.random_marks(seed, cfgs[i]["max_blocks"], p_refine=0.4, p_coarsen=0.0)
            sim.adapt(torch.from_numpy(m).cuda())
        g = np.random.default_rng(7 + i)
        sim.set_populations(w * (1 + 0.02 * (2 * g.random((cfgs[i]["max_blocks"], 64, q)) - 1)))
        return sim

    want = []
    for i in range(2):
        sim = forest(i, "f32")
        sim.step(STEPS)
        want.append(sim.populations()[sim.blocks()["level"] >= 0])
        sim.close()
    for threads, tile in ((64, 1), (64, 8), (128, 1), (128, 2), (128, 8), (256, 1), (256, 3),
                          (256, 4), (256, 5), (256, 8)):
        members = [forest(i, storage) for i in range(2)]
        batch = AmrBatch(members)
        batch.configure("persistent", threads, tile)
        batch.step(STEPS)
        batch.sync()
        for sim, ref in zip(members, want):
            got = sim.populations()[sim.blocks()["level"] >= 0]
            bound = (1 + 2 * 4 * STEPS) * u * np.linalg.norm(ref - w) / np.linalg.norm(ref)
            assert np.linalg.norm(got - ref) <= bound * np.linalg.norm(ref), (threads, tile)
        batch.close()
        for sim in members:
            sim.close()
