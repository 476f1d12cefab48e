"""Rounding error of the proposal network's gradient."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def net(w, x):
    a = [w[:1728].reshape(64, 27), w[1728:1792], w[1792:5888].reshape(64, 64), w[5888:5952],
         w[5952:6016], w[6016]]
    return torch.relu(torch.relu(x @ a[0].T + a[1]) @ a[2].T + a[3]) @ a[4] + a[5]


@pytest.mark.parametrize("n", [500, 1024])
def test_gradient_is_summed_in_few_additions(n):
    """An entry is a sum of K partial sums in FP32.  The error of K additions,
    each 0.4 u of a partial sum in the mean (u = 2^-24) that grows like the root
    of its terms, is 0.4 u sqrt(K / 2) of the entry: 1e-7 with K = 32 for 1,024
    samples, 2.7e-7 with one addition per tile of four (K = 256), to which the
    errors of the terms (dot products of 64) add some 5e-8.  Of 500 samples
    7e-8 with 16, 1.9e-7 with 125.  The bars lie between, for the mean of eight
    draws."""
    from paper_2308_08085_gb300.amr import Mlp
    total = 0.0
    for seed in range(8):
        g = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.randn(n, 27, generator=g, device="cuda")
        y = (torch.rand(n, generator=g, device="cuda") < 0.3).float()
        mlp = Mlp(torch.device("cuda"), seed=seed)
        grad, _ = mlp.grad_of(x, y, pos_weight=3.0)
        w = mlp.params.double().requires_grad_(True)
        z = net(w, x.double())
        sp = torch.nn.functional.softplus
        ref, = torch.autograd.grad((3.0 * y.double() * sp(-z) + (1 - y.double()) * sp(z)).sum(), w)
        total += float((grad.double() - ref).norm() / ref.norm()) / 8
    assert total < {500: 1.5e-7, 1024: 1.8e-7}[n], total
