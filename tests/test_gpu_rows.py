"""Edges of the kernels that read blocks by x-rows and of the rules that choose
them: chained and unchained launches of a coarse step, exports to destinations
that vector stores cannot reach, and the tile sizes of the proposal network's
gradient and inference."""
import ctypes

import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


def _cfg(dim, q, flow, interp):
    if flow == "prism":
        cfg = W.channel_cylinder(q=q, nx=32, ny=20, nz=8, side=4, cx=10, cy=10, max_levels=3,
                                 max_blocks=4000 if dim == 3 else 1200, refine_dist=0.0, dim=dim)
    else:
        cfg = W.cavity(dim=dim, q=q, n=20, ny=12, nz=8, max_levels=3,
                       max_blocks=4000 if dim == 3 else 1200)
    cfg["interp"] = interp
    return cfg


def _forest(cfg, storage, **kw):
    from paper_2308_08085_gb300 import AmrLBM
    sim = AmrLBM(cfg, storage=storage, **kw)
    for seed in (3, 4):
        m = W.random_marks(seed, cfg["max_blocks"], p_refine=0.4, p_coarsen=0.0)
        sim.adapt(torch.from_numpy(m).cuda())
    return sim


@pytest.mark.parametrize("dim,q", [(2, 9), (3, 19), (3, 27)])
@pytest.mark.parametrize("storage", ["f64", "f32", "f16"])
@pytest.mark.parametrize("flow,interp", [("cavity", "linear"), ("prism", "linear"),
                                         ("prism", "cubic")])
def test_chained_launches_equal_plain_ones(dim, q, storage, flow, interp):
    """The captured coarse step (small launches chained) and the same launches
    one by one run the same kernels on the same values: equal bit for bit."""
    if dim == 2 and storage == "f16":
        pytest.skip("16-bit storage is 3D only")
    cfg = _cfg(dim, q, flow, interp)
    a = _forest(cfg, storage, use_graphs=True)
    b = _forest(cfg, storage, use_graphs=False)
    b.restore(a.checkpoint())
    a.step(7)
    b.step(7)
    torch.cuda.synchronize()
    fa, fb = a.populations(), b.populations()
    assert np.isfinite(fa).all()
    assert np.array_equal(fa, fb)


@pytest.mark.parametrize("dim,q", [(2, 9), (3, 19)])
def test_export_to_an_unaligned_destination(dim, q):
    """A device destination aligned to 8 bytes only takes the scalar stores."""
    from paper_2308_08085_gb300 import amr
    sim = _forest(_cfg(dim, q, "prism", "linear"), "f32")
    sim.step(2)
    for what in (amr.AMR_RHO_U, amr.AMR_F):
        n = sim.field_bytes(what)
        ref = sim.fields_device(what, torch.float64)
        for skip in (1, 2, 3):
            buf = torch.full((n // 8 + 4,), -7.0, dtype=torch.float64, device="cuda")
            got = sim.lib.amr_fields(sim.h, what, ctypes.c_void_p(buf.data_ptr() + 8 * skip), n, 1)
            assert got == n
            assert torch.equal(buf[skip:skip + n // 8], ref)
            assert (buf[:skip] == -7.0).all() and (buf[skip + n // 8:] == -7.0).all()


def _net(w, x):
    a = [w[:1728].reshape(64, 27), w[1728:1792], w[1792:5888].reshape(64, 64), w[5888:5952],
         w[5952:6016], w[6016]]
    return torch.relu(torch.relu(x @ a[0].T + a[1]) @ a[2].T + a[3]) @ a[4] + a[5]


# a sample, tiles of 4 cut off, clusters of 8 CTAs cut off, the change to tiles
# of 8 (above 1216 samples), and more tiles than CTAs (above 2432)
@pytest.mark.parametrize("n", [1, 3, 5, 32, 33, 1215, 1216, 1217, 2433, 5003])
def test_gradient_tiles(n):
    """Against FP64 autograd.  A gradient entry is a sum over the samples of
    products of three dot products of up to 64 terms in FP32: relative error of
    the whole gradient within 3 x 64 x 2^-24 = 1.1e-5."""
    from paper_2308_08085_gb300.amr import Mlp
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.randn(n, 27, generator=g, device="cuda")
    y = (torch.rand(n, generator=g, device="cuda") < 0.3).float()
    mlp = Mlp(torch.device("cuda"), seed=n)
    grad, loss = mlp.grad_of(x, y, pos_weight=3.0)
    w = mlp.params.double().requires_grad_(True)
    z = _net(w, x.double())
    sp = torch.nn.functional.softplus
    ref = (3.0 * y.double() * sp(-z) + (1 - y.double()) * sp(z)).sum()
    rg, = torch.autograd.grad(ref, w)
    assert float((grad.double() - rg).norm() / rg.norm()) < 1.1e-5
    assert abs(float(loss) / float(ref) - 1) < 1.1e-5


# one sample per thread up to 38,912 samples, two above; CTAs of 64
@pytest.mark.parametrize("n", [1, 63, 64, 65, 38912, 38913, 39040])
def test_inference_tiles(n):
    """Probabilities against FP64 with the same FP16 weights: z carries the
    rounding of 64-term FP32 dot products, and a sigmoid has slope 1/4 at most."""
    from paper_2308_08085_gb300.amr import Mlp
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.randn(n, 27, generator=g, device="cuda")
    mlp = Mlp(torch.device("cuda"), seed=1)
    ref = torch.sigmoid(_net(mlp.half.double(), x.double()))
    assert float((mlp.infer(x).double() - ref).abs().max()) < 1.1e-5
