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


@pytest.mark.parametrize("prec,o,v,limit", [("ozaki", 2, 3, 202752), ("ozaki", 3, 9, 2297856), ("ozaki", 2, 17, 1775616),
                                            ("ozaki", 4, 24, 13189120), ("ozaki", 2, 65, 31162368),
                                            ("bf16x3", 2, 3, 124928), ("bf16x3", 4, 24, 6774784),
                                            ("bf16x3", 8, 64, 43974656), ("tf32", 5, 81, 58589184),
                                            ("tf32", 6, 161, 389021696)])
def test_tensor_core_energy_under_its_old_limit(te, prec, o, v, limit):
    a = cluster(o, v)
    e = limited(te, limit, lambda h: te.t_energy_triples(a, precision=prec, handle=h))
    assert torch.equal(e, te.t_energy_triples(a, precision=prec, handle=te.Handle(0)))


@pytest.mark.parametrize("o,v,limit", [(2, 8, 140288), (4, 24, 1830912), (8, 64, 33554432), (4, 72, 29360128),
                                       (16, 120, 365953024)])
def test_one_triple_under_its_old_limit(te, o, v, limit):
    a = cluster(o, v)
    e = limited(te, limit, lambda h: te.t_energy_triples(a, 1, 2, "ozaki", handle=h))
    assert torch.equal(e, te.t_energy_triples(a, 1, 2, "ozaki", handle=te.Handle(0)))


@pytest.mark.parametrize("o,v,limit", [(1, 1, 163840), (2, 8, 244736), (4, 24, 2412544), (8, 40, 15384576), (2, 65, 31358976),
                                       (3, 80, 60227584), (3, 97, 119144448), (16, 120, 540016640), (3, 201, 914358272),
                                       (4, 320, 3514826752)])
def test_exact_slice_gradient_under_its_old_limit(te, o, v, limit):
    """Less workspace sums the same slice products in other blocks (1e-8 of the
    largest entry)."""
    a = cluster(o, v)
    _, g = limited(te, limit, lambda h: te.t_energy_vjp(a, precision="ozaki", handle=h))
    _, ref = te.t_energy_vjp(a, precision="ozaki", handle=te.Handle(0))
    for n in NAMES:
        assert float((g[n] - ref[n]).abs().max()) <= 1e-8 * float(ref[n].abs().max()), n


@pytest.mark.parametrize("o,v,limit", [(1, 1, 43008), (2, 3, 80896)])
def test_exact_slice_projected_energy_under_its_old_limit(te, o, v, limit):
    a = cluster(o, v)
    cf = np.random.default_rng(v).standard_normal((o, o))
    _, e = limited(te, limit, lambda h: te.t_energy_frag(a, cf, "ozaki", handle=h, shares=True))
    _, ref = te.t_energy_frag(a, cf, "ozaki", handle=te.Handle(0), shares=True)
    assert torch.equal(e, ref)


def held(te, h):
    """Device memory in use: the handle's workspace is the only thing that moves it."""
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free


@pytest.mark.parametrize("what,prec,large,small", [
    ("energy", "ozaki", (16, 161), (16, 160)), ("energy", "ozaki", (5, 161), (4, 160)),
    ("energy", "bf16x3", (16, 257), (16, 256)), ("energy", "fp64", (10, 129), (10, 128)),
    ("vjp", "ozaki", (33, 320), (32, 320)), ("vjp", "ozaki", (18, 400), (17, 400)), ("vjp", "ozaki", (4, 201), (4, 200)),
    ("frag", "ozaki", (6, 97), (6, 96))])
def test_reserve_covers_smaller_sizes(te, what, prec, large, small):
    """Sizes across which the larger cluster needs less."""
    h = te.Handle(0)
    kinds = {k: k == what for k in ("energy", "vjp", "frag")}
    h.reserve(*large, prec, **kinds)
    before = held(te, h)
    h.reserve(*small, prec, **kinds)
    assert held(te, h) == before


@pytest.mark.parametrize("prec", ["fp64", "ozaki"])
def test_smaller_energy_is_capturable_after_reserve(te, prec):
    h = te.Handle(0)
    h.reserve(4, 161, prec)
    before = held(te, h)
    a = cluster(4, 160)
    grown = held(te, h) - before  # the inputs
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        out = te.t_energy(a, prec, handle=h, stream=s)
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert float(out) == float(te.t_energy(a, prec, handle=te.Handle(0)))
    h.sync()
    assert grown >= 0


def test_smaller_gradient_allocates_nothing_after_reserve(te):
    h = te.Handle(0)
    h.reserve(4, 201, "ozaki", energy=False, vjp=True)
    a = cluster(4, 200)
    h0 = te.Handle(0)
    te.t_energy_vjp(a, precision="ozaki", handle=h0)  # torch then has the gradients' memory in its cache
    h0.sync()
    h0.close()
    before = held(te, h)
    te.t_energy_vjp(a, precision="ozaki", handle=h)
    h.sync()
    assert held(te, h) == before


@pytest.fixture
def little_memory(te):
    """Leaves `room` bytes of the device free, beside what torch has cached."""
    kept = []

    def fill(room):
        torch.cuda.synchronize()
        kept.append(torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda"))

    yield fill
    kept.clear()
    torch.cuda.empty_cache()


def test_gradients_and_reservation_where_only_the_lean_form_fits(te, little_memory):
    """nocc=8 nvir=64: 49 MB do (the limit above); what the usual form takes is
    measured here."""
    o, v = 8, 64
    a = cluster(o, v)
    h = te.Handle(0)
    before = held(te, h)
    h.reserve(o, v, "ozaki", energy=False, vjp=True)
    usual = held(te, h) - before
    h.close()
    room = 64 << 20
    assert usual > 2 * room
    ref, g = te.t_energy_vjp(a, precision="ozaki", handle=te.Handle(0))  # and torch's cache for the gradients
    g = {n: x.cpu() for n, x in g.items()}
    h1, h2 = te.Handle(0), te.Handle(0)
    e, grads = te.t_energy_vjp_batched([a], precision="fp64", handle=te.Handle(0))
    del e, grads
    little_memory(room)
    e, grads = te.t_energy_vjp_batched([a], precision="ozaki", handle=h1)
    h1.sync()
    assert abs(float(e[0]) - float(ref)) <= 1e-12 * abs(float(ref))
    for n in NAMES:
        assert float((grads[0][n].cpu() - g[n]).abs().max()) <= 1e-8 * float(g[n].abs().max())
    first = held(te, h1)
    del e, grads
    te.t_energy_vjp_batched([a], precision="ozaki", handle=h1)  # the same form, nothing allocated
    h1.sync()
    assert held(te, h1) == first
    h1.close()
    h2.reserve(o, v, "ozaki", energy=False, vjp=True)
    first = held(te, h2)
    te.t_energy_vjp(a, precision="ozaki", handle=h2)
    h2.sync()
    assert held(te, h2) == first


@pytest.mark.parametrize("o,v,naux,prec,limit", [(2, 10, 50, "fp64", 76288), (2, 10, 50, "ozaki", 84736)])
def test_mp2_under_its_old_limit(te, o, v, naux, prec, limit):
    c = tegen.mp2_inputs(o, v, naux, 5)
    out = limited(te, limit, lambda h: te.mp2_bno_batched([c], prec, handle=h))[0]
    ref = te.mp2_bno_batched([c], prec, handle=te.Handle(0))[0]
    for n in ref:
        assert torch.equal(out[n], ref[n]), n


def test_mp2_groups_of_many_clusters(te):
    """More than one group of the eigensolver, sizes that grow and shrink: the
    tridiagonal forms and the transient arrays of other clusters share memory."""
    sizes = [(1 + x % 3, 1 + (7 * x) % 23) for x in range(67)] + [(3, 40)]
    cs = [tegen.mp2_inputs(o, v, 2 * (o + v), x) for x, (o, v) in enumerate(sizes)]
    out = te.mp2_bno_batched(cs, "fp64", handle=te.Handle(0))
    for x in (0, 1, 30, 31, 32, 33, 63, 64, 66, 67):
        one = te.mp2_bno_batched([cs[x]], "fp64", handle=te.Handle(0))[0]
        for n in one:
            assert torch.equal(out[x][n], one[n]), (x, n)
