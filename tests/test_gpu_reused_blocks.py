"""Blocks whose IDs were used before, next to a solid: the children of fluid
blocks are removed, their IDs return as partly solid blocks of a three-level
forest whose coarse-fine interface touches the prism.  Solid cells hold the rest
state in whatever the interpolation reads, also in the buffer of the second
substep, against the oracle."""
import numpy as np
import pytest

import workloads as W
from cellwise import assert_cells, oracle_classes
from oracle.lattice import equilibrium
from oracle.solver import ForestLBM

torch = pytest.importorskip("torch")


def config(dim, q, interp):
    """A prism of one root cell's width centred on a root cell's edge: its sides
    lie in the middle of level-0 cells, on cell faces of level 1, inside the
    quadrant of parent cells that a child is interpolated from."""
    cfg = W.channel_cylinder(dim=dim, q=q, nx=24, ny=20, nz=4, side=1, cx=10, cy=10, re=10.0,
                             max_levels=3, max_blocks=600, refine_dist=0.0)
    cfg["interp"] = interp
    return cfg


def marks(mesh, level, inside, value):
    """`value` on the blocks of a level whose corner is `inside`."""
    m = np.zeros(mesh.cap, np.int8)
    for b in mesh.active_ids():
        if mesh.level[b] == level and inside(mesh.X[b]):
            m[b] = value
    return m


def randomize(ref, seed):
    ids = np.array(ref.mesh.active_ids())
    n = len(ids) * ref.m
    rho, u = W.random_macro(seed, n, ref.dim)
    f = (equilibrium(ref.vs, rho, u) + W.random_noise(seed + 1, (n, ref.vs.q), 1e-3)).reshape(
        len(ids), ref.m, ref.vs.q)
    f[ref.solid[ids]] = ref.rest
    ref.f[ids] = f


def reuse(ref, others):
    """The sequence on the oracle and every instance of `others`."""
    def far(x):
        return x[0] >= 16

    def near(x):
        return 4 <= x[0] < 16 and 4 <= x[1] < 16

    def left(x):
        return x[0] < 10 and 6 <= x[1] < 14

    def adapt(m):
        ref.adapt(m)
        for sim in others:
            sim.adapt(torch.from_numpy(m).cuda())

    def step(n):
        ref.step(n)
        for sim in others:
            sim.step(n)

    adapt(marks(ref.mesh, 0, far, 1))
    old = set(ref.mesh.id_sets[1])
    randomize(ref, 5)
    for sim in others:
        sim.set_populations(ref.f)
    step(2)                                   # both buffers hold fluid values
    adapt(marks(ref.mesh, 0, far, -1))
    assert not ref.mesh.id_sets[1]
    adapt(marks(ref.mesh, 0, near, 1))
    adapt(marks(ref.mesh, 1, left, 1))
    # partly solid exchanging parents of level 1 with IDs that were fluid
    parents = [b for b in ref.mesh.parent_list(1)
               if b in old and ref.solid[b].any() and not ref.solid[b].all()]
    assert parents
    step(3)
    ref.sync()


@pytest.mark.parametrize("dim,q", [(2, 9), (3, 19)])
def test_the_sequence_reuses_partly_solid_parents(dim, q):
    reuse(ForestLBM(config(dim, q, "linear")), [])


@pytest.mark.gpu
@pytest.mark.parametrize("dim,q", [(2, 9), (3, 19), (3, 27)])
@pytest.mark.parametrize("interp", ["linear", "cubic"])
def test_reused_blocks_at_a_solid(dim, q, interp):
    """FP64 within the bars of the other parity tests (1e-12 relative L2, 1e-10
    per cell), as a graph and launch by launch; FP16 and BF16 storage (the
    solid's shifted rest state is zero) within the rounding of its stores."""
    from paper_2308_08085_gb300 import AmrLBM
    cfg = config(dim, q, interp)
    ref = ForestLBM(cfg)
    small = [] if dim == 2 else [("f16", 2.0 ** -11), ("bf16", 2.0 ** -8)]
    sims = [AmrLBM(cfg, storage="f64", use_graphs=g) for g in (False, True)]
    sims += [AmrLBM(cfg, storage=s) for s, _ in small]
    reuse(ref, sims)
    ids = ref.mesh.active_ids()
    for sim in sims:
        sim.rho_u()                           # runs the level synchronisation
    for sim in sims[:2]:
        got = sim.populations()[ids]
        assert np.linalg.norm(got - ref.f[ids]) <= 1e-12 * np.linalg.norm(ref.f[ids])
        assert_cells(got, ref.f[ids], oracle_classes(ref.mesh, ids), ref.vs.w, "f64")
    g = ref.f[ids] - ref.vs.w
    for sim, (_, u) in zip(sims[2:], small):
        # a value goes through the import, then per substep of the finest level
        # (4 a coarse step, 5 coarse steps) a collision and an exchange, and the
        # four adaptations and the read-back: each rounds f - w by u at most
        got = sim.populations()[ids]
        bound = (1 + 2 * 4 * 5 + 5) * u * np.linalg.norm(g) / np.linalg.norm(ref.f[ids])
        assert np.linalg.norm(got - ref.f[ids]) <= bound * np.linalg.norm(ref.f[ids])
