"""Launches of a captured coarse step that are programmatic dependents of the
one before (chained): the source keeps the rules that make them safe, and large
and small launches next to one another give the results of plain launches."""
import os
import re

import numpy as np
import pytest

import workloads as W

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2308_08085_gb300", "csrc")


def functions():
    """{name: (parameters, body)} of the device functions and kernels."""
    out = {}
    for name in ("lattice.cuh", "collide_stream.cuh", "lbm_kernels.cuh"):
        s = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        for m in re.finditer(r"(?:__device__ (?:__forceinline__|__noinline__)|__global__)[^;{}=]*?"
                             r"\b(\w+)\(((?:[^(){};]|\([^()]*\))*)\)\s*\{", s):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(s[i], 0)
                i += 1
            old = out.get(m.group(1), ("", ""))
            out[m.group(1)] = (old[0] + "," + m.group(2), old[1] + s[m.end():i - 1])
    return out


def test_population_pointers_of_chained_kernels_are_plain():
    """A dependent kernel is resident while its predecessor writes: neither it
    nor what it calls may promise that populations are read-only or unaliased."""
    f = functions()
    chained = {"k_collide_stream", "k_average", "k_average_groups"}
    assert {n for n in f if n.startswith("k_") and "chain_wait();" in f[n][1]} == chained
    reach, todo = set(), list(chained)
    while todo:
        n = todo.pop()
        if n not in reach:
            reach.add(n)
            todo += [c for c in f if re.search(r"\b%s\s*[<(]" % c, f[n][1])]
    assert {"step_row", "gather_row", "interp_rows", "average_lanes"} <= reach
    bad = [(n, p.strip()) for n in sorted(reach) for p in f[n][0].split(",")
           if re.search(r"\bT\s*\*\s*__restrict__", p)]
    assert not bad


def test_every_chained_launch_waits():
    """A kernel launched by launch_chained calls chain_wait, before any access
    to populations: they are not named above the wait."""
    f = functions()
    src = open(os.path.join(CSRC, "lbm_kernels.cuh")).read()
    launched = set(re.findall(r"launch_chained\(\s*(?:solid \? )?(k_\w+)", src))
    assert launched == {"k_collide_stream", "k_average", "k_average_groups"}
    for n in launched:
        pops = re.findall(r"\bT\s*\*\s*(\w+)", f[n][0])
        before = f[n][1].rpartition("chain_wait();")[0]
        assert pops and not [p for p in pops if re.search(r"\b%s\b" % p, before)]
        # a thread without work waits as well
        for part in before.split("return;")[:-1]:
            assert "chain_wait();" in part


def large_and_small(interp, storage, **kw):
    """Three levels: 128 / 384 active blocks, 8192 on the finest (chained up to
    2048 blocks)."""
    import torch
    from paper_2308_08085_gb300 import AmrLBM
    cfg = W.cavity(dim=3, q=19, n=32, ny=32, nz=16, max_levels=3, max_blocks=10000)
    cfg["interp"] = interp
    sim = AmrLBM(cfg, storage=storage, **kw)
    for level, reach in ((0, 0.6), (1, 0.5)):
        b, x = sim.blocks(), sim.coords()[:, 0] / 32
        marks = ((b["level"] == level) & (x < reach)).astype(np.int8)
        sim.adapt(torch.from_numpy(marks).cuda())
    n = sim.counts()["n_active"]
    assert n[0] < 2048 and n[1] < 2048 < n[2], n
    return sim


@pytest.mark.gpu
@pytest.mark.parametrize("storage", ["f32", "f64", "f16"])
@pytest.mark.parametrize("interp", ["linear", "cubic"])
def test_large_and_small_launches(interp, storage):
    """Chained launches after large plain ones and before them, in a single
    instance and in a batch's branches (which take linear interpolation only),
    against plain launches: bit for bit."""
    import torch
    from paper_2308_08085_gb300 import AmrBatch
    a = large_and_small(interp, storage, use_graphs=True)
    plain = large_and_small(interp, storage, use_graphs=False)
    members = [large_and_small(interp, storage) for _ in range(2 if interp == "linear" else 0)]
    a.step(3)
    image = a.checkpoint()
    for sim in [plain] + members:
        sim.restore(image)
    batch = AmrBatch(members) if members else None
    if batch:
        batch.configure("members")
    for n in (1, 8, 15):
        a.step(n)
        plain.step(n)
        if batch:
            batch.step(n)
        torch.cuda.synchronize()
        want = plain.populations()
        assert np.isfinite(want).all()
        for sim in [a] + members:
            assert np.array_equal(sim.populations(), want)
    if batch:
        batch.close()
