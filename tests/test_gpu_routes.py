"""Sizes at which the routes inside one entry point meet: edges of the tiles, the
least workspace a call accepts, and orders at which the eigensolver changes.

Tolerances: exact-slice gradients carry the bar of 1e-6 of a tensor's largest
entry.  The same gradient with less workspace sums the same exact slice products
in blocks of another size: their third accumulator (2^-14 of the operands' scale)
rounds at 2^-24, 2^-38 = 4e-12 of a scale that may lie 1e3 above the result, so
1e-8.  Projected shares have the same blocks either way and differ in FP32-pair
sums only (2^-48 per term, some thousand terms): 1e-10 of the largest.  A
Householder reduction and bisection are backward stable: order times 2^-53 times a
small constant, 1e-12 of the norm up to order 520 as for any solver here."""
import numpy as np
import pytest
import torch

import tegen
from oracle import t_energy as O
from gpu_common import need_gpu, shuffled

pytestmark = pytest.mark.gpu

NAMES = ("eps_o", "eps_v", "ovvv", "ooov", "ovov", "t1", "t2")


@pytest.fixture(scope="module")
def te():
    return need_gpu()


def dev(arrs):
    return {n: torch.as_tensor(np.ascontiguousarray(arrs[n])).cuda() for n in NAMES}


def cluster(o, v, seed):
    arrs = shuffled(tegen.make_cluster(o, v, 4 * (o + v), seed).arrays(), seed)
    arrs["t1"] = arrs["t1"] * 50.0
    return arrs


def least_workspace(te, call):
    """call(handle) under the smallest limit (within a fifth) that it accepts."""
    limit = 1 << 20
    while True:
        h = te.Handle(0)
        h.set_workspace_limit(int(limit))
        try:
            out = call(h)
            h.sync()
            return out
        except te.TEnergyError as err:
            assert "limit" in str(err)
        limit *= 1.2


@pytest.mark.parametrize("v", [1, 8, 9, 31, 32, 33, 63, 64, 65, 97])
def test_float64_energy_at_tile_edges(te, v):
    arrs = cluster(3, v, 40 + v)
    ref = float(O.t_energy(O.inputs(**arrs)))
    assert abs(float(te.t_energy(dev(arrs), "fp64")) - ref) <= 1e-11 * abs(ref) + 1e-15


@pytest.mark.parametrize("o,v", [(2, 32), (3, 33), (4, 64), (2, 65), (2, 96), (5, 97), (2, 128), (2, 129), (2, 201)])
def test_gradient_routes(te, o, v):
    """Exact slices against float64, and the least workspace against plenty
    (transposes formed triple by triple, batches of one)."""
    a = dev(cluster(o, v, 60 + v))
    _, g64 = te.t_energy_vjp(a, precision="fp64")
    _, g = te.t_energy_vjp(a, precision="ozaki")
    _, low = least_workspace(te, lambda h: te.t_energy_vjp(a, precision="ozaki", handle=h))
    for n in NAMES:
        top = float(g64[n].abs().max())
        assert float((g[n] - g64[n]).abs().max()) <= 1e-6 * top, n
        assert float((g[n] - low[n]).abs().max()) <= 1e-8 * top, n


@pytest.mark.parametrize("o,v", [(2, 17), (4, 64), (4, 65)])
def test_least_workspace_of_the_energies(te, o, v):
    """Fewer G slots: the same shares; projected energies one triple at a time."""
    a = dev(cluster(o, v, 80 + v))
    full = te.t_energy_triples(a, precision="ozaki")
    low = least_workspace(te, lambda h: te.t_energy_triples(a, precision="ozaki", handle=h))
    assert torch.equal(full, low)
    cf = np.random.default_rng(v).standard_normal((o, o))
    _, full = te.t_energy_frag(a, cf, "ozaki", shares=True)
    _, low = least_workspace(te, lambda h: te.t_energy_frag(a, cf, "ozaki", handle=h, shares=True))
    assert float((full - low).abs().max()) <= 1e-10 * float(full.abs().max())


@pytest.mark.parametrize("o,v,naux", [(1, 1, 1), (2, 2, 7), (5, 34, 33), (3, 167, 8), (2, 168, 9), (1, 520, 4)])
@pytest.mark.parametrize("scale", [1.0, 0.0])
def test_populations(te, o, v, naux, scale):
    """Orders around the shared-memory and thread counts; scale 0: gamma_vv = 0 and
    gamma_oo = 2."""
    eps_o, eps_v, B = tegen.mp2_inputs(o, v, naux, 7)
    out = te.mp2_bno_batched([(eps_o, eps_v, B * scale)], "fp64")[0]
    for gn, pn in (("gamma_oo", "pop_o"), ("gamma_vv", "pop_v")):
        g, p = out[gn].cpu().numpy(), out[pn].cpu().numpy()
        assert np.all(np.diff(p) >= 0.0)
        assert np.abs(p - np.linalg.eigvalsh(0.5 * (g + g.T))).max() <= 1e-12 * np.abs(g).max() + 1e-300


@pytest.mark.parametrize("o,v,naux", [(1, 3, 1), (2, 33, 7), (2, 64, 8), (2, 65, 31), (3, 43, 33), (2, 20, 1025)])
def test_exact_slice_mp2_integrals_at_edges(te, o, v, naux):
    """Rows, columns and auxiliary indices off the tiles (128, 128, 32; blocks of 1024)."""
    c = tegen.mp2_inputs(o, v, naux, 11)
    a, b = te.mp2_bno_batched([c], "fp64")[0], te.mp2_bno_batched([c], "ozaki")[0]
    for n in ("t2", "gamma_oo", "gamma_vv"):
        assert float((a[n] - b[n]).abs().max()) <= 1e-7 * float(a[n].abs().max()), n
