"""Refinement marks are integers that rest on thresholds of computed values, so
the values behind them are kept bit for bit: the block summaries, the marks of
the learned proposal with the threshold on the probability of a leaf, the marks
of the vorticity criterion and the synchronised populations they are read from,
against golden/marks.npz.  The golden values were computed by the kernels with a
thread per cell, whose sums run in cell order:

    python tests/test_gpu_marks.py OUT.npz      # writes the values of this build
"""
import hashlib
import os
import sys

import numpy as np
import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "marks.npz")
CASES = [("cavity", 19, "f32", "linear"), ("prism", 27, "f32", "linear"),
         ("cavity", 27, "f64", "cubic"), ("prism", 19, "f64", "linear"),
         ("prism", 19, "bf16", "linear"), ("cavity", 27, "f16", "cubic")]


def values(flow, q, storage, interp):
    """What the test compares: a seeded state on a three-level forest."""
    from oracle.lattice import VelocitySet
    from paper_2308_08085_gb300 import AmrLBM, Mlp
    if flow == "prism":
        cfg = W.channel_cylinder(q=q, nx=32, ny=20, nz=8, side=4, cx=10, cy=10, max_levels=3,
                                 max_blocks=1200, refine_dist=0.0)
    else:
        cfg = W.cavity(dim=3, q=q, n=20, ny=12, nz=8, max_levels=3, max_blocks=1200)
    cfg["interp"] = interp
    sim = AmrLBM(cfg, storage=storage)
    for seed in (3, 4):
        marks = W.random_marks(seed, cfg["max_blocks"], p_refine=0.2, p_coarsen=0.0)
        sim.adapt(torch.from_numpy(marks).cuda())
    g = np.random.default_rng(17)
    w = VelocitySet(3, q).w
    f = w * (1.0 + 0.02 * (2.0 * g.random((cfg["max_blocks"], 64, q)) - 1.0))
    sim.set_populations(f)
    net = Mlp(torch.device("cuda", 0), seed=1)
    half = ((2.0 * g.random(net.n) - 1.0) * 0.2).astype(np.float16)
    net.half.copy_(torch.from_numpy(half))
    out = {"criterion": sim.criterion_marks().cpu().numpy()}
    feat = sim.features()
    b = sim.blocks()
    out["features"] = feat.cpu().numpy()[b["level"] >= 0]
    prob = net.infer(feat).cpu().numpy()[b["status"] == 1]
    for i, part in enumerate((0.25, 0.5, 0.75)):
        at = np.sort(prob)[int(part * len(prob))]     # the probability of a leaf
        out["threshold%d" % i] = at
        out["marks%d" % i] = sim.propose_marks(net.half, float(at)).cpu().numpy()
        out["alone%d" % i] = sim.propose_marks(net.half, float(at), False).cpu().numpy()
    out["populations"] = np.array(hashlib.sha256(sim.populations().tobytes()).hexdigest())
    sim.close()
    return out


@pytest.mark.parametrize("case", CASES, ids=["-".join(map(str, c)) for c in CASES])
def test_marks_and_what_they_rest_on(case):
    from paper_2308_08085_gb300 import build as b
    b.build()
    want = np.load(GOLDEN)
    got = values(*case)
    for k, v in got.items():
        assert np.array_equal(v, want["-".join(map(str, case)) + "." + k]), k


if __name__ == "__main__":
    np.savez_compressed(sys.argv[1], **{"-".join(map(str, c)) + "." + k: v
                                        for c in CASES for k, v in values(*c).items()})
