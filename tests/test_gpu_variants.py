"""amr_config.kernel_variant takes any integer: values without a kernel of their
own take the default one."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,q", [(2, 9), (3, 19)])
def test_any_variant_steps(dim, q):
    """Bit for bit the step of the default, which moves a cavity off rest."""
    from paper_2308_08085_gb300 import AmrLBM, build as b
    b.build()
    cfg = W.cavity(dim=dim, q=q, n=16, max_levels=1)
    got = {}
    for variant in (0, -1, 6, -2 ** 31, 2 ** 31 - 1):
        sim = AmrLBM(cfg, storage="f32", kernel_variant=variant)
        rest = sim.populations()
        sim.step(3)
        got[variant] = sim.populations()
        assert not np.array_equal(got[variant], rest)
        assert np.array_equal(got[variant], got[0])
        sim.close()
