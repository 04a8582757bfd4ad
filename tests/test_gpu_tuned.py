"""The configurations that the autotuners find, run: the named workloads with
the returned configuration passed on, and an uneven plan built from the tuned
table."""
import numpy as np
import pytest

import paper_2410_22575_gb300 as cf
from paper_2410_22575_gb300 import workloads as W

from gpu_helpers import BOUND, Dev, hvp_err
from test_gpu_ragged import DevRagged

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [cf.FP32_COMP, cf.FP64])
@pytest.mark.parametrize("fn,n,batch", [(W.ROSENBROCK, 16, 4096), (W.ACKLEY, 64, 4096), (W.FLETCHER_POWELL, 32, 1024),
                                        (W.ROSENBROCK, 130, 64)])
def test_tuned_configuration(prec, fn, n, batch):
    import torch

    d = Dev(W.make_batch(fn, n, batch, seed=n), prec)
    cfg = cf.chessfad_autotune_hvp(fn, n, batch, d.x, d.v, torch.empty_like(d.x), d.params, prec)
    assert cfg.csize in (1, 2, 4, 8, 16, 32)
    e = hvp_err(d, d.hvp(cfg=cfg))
    assert e.max() <= BOUND[prec], (cfg.as_dict(), e.max())


@pytest.mark.parametrize("prec", [cf.FP32_COMP, cf.FP64])
def test_uneven_plan_of_the_tuned_table(prec):
    """The plan's groups have the tuned chunk sizes, its tiles are the dense
    ones, and every request meets the bound against the oracle."""
    import torch

    rg = W.make_ragged(nreq=900, seed=31, nmax=200)
    d = DevRagged(rg, prec, 16)
    reqs = cf.requests(rg.fns, rg.ns, rg.offs, rg.eoffs)
    cf.chessfad_ragged_autotune(reqs, prec, d.x, d.v, d.out, d.params, d.plan.workspace, d.plan.workspace.numel())
    plan = cf.RaggedPlan(reqs, prec, tuned=True)
    groups = sorted({(int(f), int(n)) for f, n in zip(rg.fns, rg.ns)})
    chunks = set()
    for f, n in groups:
        c = cf.chessfad_ragged_plan_group_config(plan.handle, f, n)[0]
        assert c == cf.chessfad_ragged_tuned_config(prec, f, n)[0]
        chunks.add(c)
    # a group has a tile of its own: 256 rows at most, of one size
    assert plan.info["ntiles"] >= len(groups) and chunks <= {8, 16}
    d.out.fill_(float("nan"))
    plan.run(d.x, d.v, d.out, d.params)
    torch.cuda.synchronize()
    first = d.out.double().cpu().numpy()
    e = d.errors(first)
    assert e.max() <= BOUND[prec], e.max()
    plan.run(d.x, d.v, d.out, d.params)
    assert np.array_equal(first, d.out.double().cpu().numpy())
    plan.close()
