"""The workspace contract: a limit (te_set_workspace_limit) that once admitted a
call still does, with the same result, and what te_reserve sets aside serves every
smaller call.

The limits below are what each call needed, to 0.2% above, when it had one form
only; a call that has since grown for speed runs in a smaller form under them."""
import numpy as np
import pytest
import torch

import tegen
from gpu_common import need_gpu

pytestmark = pytest.mark.gpu

NAMES = ("eps_o", "eps_v", "ovvv", "ooov", "ovov", "t1", "t2")


@pytest.fixture(scope="module")
def te():
    return need_gpu()


def dev(arrs):
    return {n: torch.as_tensor(np.ascontiguousarray(arrs[n])).cuda() for n in NAMES}


def cluster(o, v):
    """Inputs whose values do not matter here, drawn on the device."""
    g = torch.Generator(device="cuda").manual_seed(o * 1000 + v)
    r = lambda *shape: torch.randn(shape, dtype=torch.float64, device="cuda", generator=g)  # noqa: E731
    t2 = 0.01 * r(o, o, v, v)
    return dict(eps_o=-1.0 - torch.rand(o, dtype=torch.float64, device="cuda", generator=g),
                eps_v=1.0 + torch.rand(v, dtype=torch.float64, device="cuda", generator=g),
                ovvv=0.1 * r(o, v, v, v), ooov=0.1 * r(o, o, o, v), ovov=0.1 * r(o, v, o, v), t1=0.01 * r(o, v),
                t2=0.5 * (t2 + t2.transpose(0, 1).transpose(2, 3)))


def limited(te, limit, call):
    h = te.Handle(0)
    h.set_workspace_limit(limit)
    out = call(h)
    h.sync()
    return out


@pytest.mark.parametrize("o,v,limit", [(8, 40, 27951104), (8, 64, 48562176), (4, 72, 28246016), (3, 80, 37814272),
                                       (14, 96, 73531392), (3, 128, 52756480)])
def test_float64_energy_under_its_old_limit(te, o, v, limit):
    a = cluster(o, v)
    e = limited(te, limit, lambda h: te.t_energy(a, "fp64", handle=h))
    assert float(e) == float(te.t_energy(a, "fp64", handle=te.Handle(0)))


def test_float64_batch_under_its_old_limit(te):
    a = [cluster(o, 8 * o) for o in (4, 5, 6)]
    e = limited(te, 32538624, lambda h: te.t_energy_batched(a, "fp64", handle=h))
    assert torch.equal(e, te.t_energy_batched(a, "fp64", handle=te.Handle(0)))
