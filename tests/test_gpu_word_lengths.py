"""What the exact-slice modes hold beside the operands' slices.

Inputs that are integers of at most 14 bits fill two 7-bit slices: every slice
product and every sum of them below 2^24 units of its level is exact, so the
contraction is exact and what separates a result from the exact one is the word
length of what is kept afterwards."""
import numpy as np
import pytest
import torch

import tegen
from gpu_common import need_gpu

pytestmark = pytest.mark.gpu

P6 = (((0, 1, 2), (0, 1, 2)), ((1, 2, 0), (2, 0, 1)), ((2, 0, 1), (1, 2, 0)),
      ((0, 2, 1), (0, 2, 1)), ((2, 1, 0), (2, 1, 0)), ((1, 0, 2), (1, 0, 2)))


@pytest.fixture(scope="module")
def te():
    return need_gpu()


def dev(arrs):
    return {n: torch.as_tensor(np.ascontiguousarray(x)).cuda() for n, x in arrs.items()}


def integers(o, v, seed):
    """Integrals and amplitudes +-(8000 + (-8 .. 8)): W~ is a 36-bit integer, nearly
    the same in all permutations of an orbit; R leaves 2^-15 of it.  No Y."""
    rng = np.random.default_rng(seed)
    n = lambda *shape: 8000.0 + rng.integers(-8, 9, shape)  # noqa: E731
    t2 = n(o, o, v, v)
    lower = np.arange(o)[:, None] > np.arange(o)
    t2[lower] = np.swapaxes(np.swapaxes(t2, 0, 1), 2, 3)[lower]
    base = tegen.make_cluster(o, v, 4 * (o + v), seed).arrays()
    return dict(eps_o=base["eps_o"], eps_v=base["eps_v"], ovvv=n(o, v, v, v), ooov=-n(o, o, o, v),
                ovov=np.zeros((o, v, o, v)), t1=np.zeros((o, v)), t2=t2)


def exact_shares(a):
    """Integer W~ and R, extended precision for the rest; sum R = 0 over an orbit,
    so W~ less a constant serves."""
    I = {k: a[k].astype(np.int64) for k in ("ovvv", "ooov", "t2")}  # noqa: E741
    eo, ev = a["eps_o"].astype(np.longdouble), a["eps_v"].astype(np.longdouble)
    out = []
    for t in [(i, j, k) for i in range(len(eo)) for j in range(i + 1) for k in range(j + 1) if not i == j == k]:
        W = 0
        for occ, vir in P6:
            p, q, r = (t[n] for n in occ)
            W = W + (np.einsum("abd,cd->abc", I["ovvv"][p], I["t2"][r, q])
                     - np.einsum("la,lbc->abc", I["ooov"][q, :, p], I["t2"][:, r])).transpose(vir)
        R = (4 * W + W.transpose(1, 2, 0) + W.transpose(2, 0, 1)
             - 2 * (W.transpose(2, 1, 0) + W.transpose(0, 2, 1) + W.transpose(1, 0, 2)))
        D = eo[list(t)].sum() - ev[:, None, None] - ev[None, :, None] - ev[None, None, :]
        m = (W - W[0, 0, 0]).astype(np.longdouble)
        out.append((m * R.astype(np.longdouble) / D).sum() * (1 if len(set(t)) == 2 else 2))
    return np.array(out)


# The differences of W~ and their products are integers that pairs hold exactly; 1/D
# comes from one Newton step on an FP32 seed, (2^-24)^2 = 4e-15, the float64 sums add 1e-15.
BAR = 2e-14


@pytest.mark.parametrize("v", [9, 33, 48, 64])
def test_energy_epilogue_where_most_of_w_cancels(te, v):
    a = integers(3, v, v)
    e = te.t_energy_triples(dev(a), precision="ozaki").cpu().numpy()
    ref = exact_shares(a)
    assert float(np.abs((e - ref) / ref).max()) <= BAR


@pytest.mark.parametrize("v", [65, 72, 79, 80])
def test_g_keeps_an_fp32_low_word_up_to_80_columns(te, v):
    """The low word of G has 10 bits here: BF16 would cut it to units of 2 to 4."""
    a = integers(3, v, v)
    e = te.t_energy_triples(dev(a), precision="ozaki").cpu().numpy()
    ref = exact_shares(a)
    assert float(np.abs((e - ref) / ref).max()) <= BAR


def test_g_formats_in_one_batch(te):
    """Members whose tiles, accumulator sets and low words differ: the shares of a
    member do not depend on the others, nor on the order of its triples."""
    a = [dev(integers(2, v, v)) for v in (96, 64, 81, 72, 65, 80, 33)]
    e = te.t_energy_batched(a, "ozaki")
    one = torch.stack([te.t_energy(x, "ozaki") for x in a])
    assert float(((e - one) / one).abs().max()) <= BAR


# Random integers of 14 bits: nothing cancels, and every product of the contraction,
# also with operands projected by 0 / 1 matrices, is exact.
def random_integers(o, v, seed, **more):
    rng = np.random.default_rng(seed)
    n = lambda *shape: rng.integers(-8000, 8001, shape).astype(float)  # noqa: E731
    t2 = n(o, o, v, v)
    lower = np.arange(o)[:, None] > np.arange(o)
    t2[lower] = np.swapaxes(np.swapaxes(t2, 0, 1), 2, 3)[lower]
    base = tegen.make_cluster(o, v, 4 * (o + v), seed).arrays()
    return dict(dict(eps_o=base["eps_o"], eps_v=base["eps_v"], ovvv=n(o, v, v, v), ooov=n(o, o, o, v),
                     ovov=n(o, v, o, v), t1=n(o, v), t2=t2), **more)


@pytest.mark.parametrize("v", [8, 17, 33])
def test_projected_energy_with_a_gap_of_1e_7(te, v):
    """D is a difference of orbital energies near 0.5 that leaves 3e-7: float64
    orders of summation agree to rounding, 1e-16 per term of some v^3 / 6, where a
    word of 48 bits would leave 1e-8 in 1 / D."""
    rng = np.random.default_rng(v)
    a = dev(random_integers(3, v, v, eps_o=-0.5 - 1e-7 * rng.random(3), eps_v=-0.5 + 1e-7 * (1.0 + rng.random(v))))
    for cf in (np.eye(3), np.diag([1.0, 0.0, 1.0])):
        _, e = te.t_energy_frag(a, cf, "ozaki", shares=True)
        _, ref = te.t_energy_frag(a, cf, "fp64", shares=True)
        assert float((e - ref).abs().max()) <= 1e-13 * float(ref.abs().max())


@pytest.mark.parametrize("o,v", [(3, 12), (4, 33), (2, 201)])
def test_gradient_of_decayed_integrals(te, o, v):
    """W~ is 2^-80 of Y (integrals and amplitudes between distant orbitals): dY, and
    with it d ovov and d t1, is a product with W~ alone.  The bar is the gradients'
    1e-6 of a tensor's largest entry."""
    a = tegen.make_cluster(o, v, 4 * (o + v), v).arrays()
    for n in ("ovvv", "ooov", "t2"):
        a[n] = a[n] * 2.0 ** -40
    a["t1"] = a["t1"] * 50.0
    a = dev(a)
    ref, g64 = te.t_energy_vjp(a, precision="fp64")
    e, g = te.t_energy_vjp(a, precision="ozaki")
    assert abs(float(e) - float(ref)) <= 1e-6 * abs(float(ref))
    for n in g:
        top = float(g64[n].abs().max())
        assert top > 0.0 and float((g[n] - g64[n]).abs().max()) <= 1e-6 * top, n


@pytest.mark.parametrize("v", [8, 17, 33])
def test_projected_energy_of_decayed_integrals(te, v):
    a = tegen.make_cluster(3, v, 4 * (3 + v), v).arrays()
    for n in ("ovvv", "ooov", "t2"):
        a[n] = a[n] * 2.0 ** -40
    a = dev(a)
    _, e = te.t_energy_frag(a, np.eye(3), "ozaki", shares=True)
    _, ref = te.t_energy_frag(a, np.eye(3), "fp64", shares=True)
    assert float((e - ref).abs().max()) <= 1e-6 * float(ref.abs().max())


@pytest.mark.parametrize("naux", [64, 1024, 2048, 5000])
@pytest.mark.parametrize("low", [0.3, -1.0])
def test_mp2_integrals_against_their_slices(te, naux, low):
    """(ia|jb) of exact slices less the sum of the slice products that are kept.  The
    level-0/1 sums are exact; the third accumulator loses at most half a unit on
    average whenever an MMA adds to it: 56 times per 128 auxiliary functions (8 steps of
    16, seven products of levels 2 and 3), a unit of 2^-34 (squares of the second slices,
    64^2 / 3 on average, make its sum 2^-10.6 on the diagonal)."""
    o, v = 2, 9
    B = np.random.default_rng(naux).uniform(low, 1.0, (naux, o, v))
    eo, ev = np.array([-1.0, -0.5]), np.linspace(0.5, 2.0, v)
    t2 = te.mp2_bno_batched([(eo, ev, B)], "ozaki")[0]["t2"].cpu().numpy()
    D = ev[:, None] + ev[None, :] - eo[:, None, None, None] - eo[:, None, None]
    rest, m, ref = B.reshape(naux, o * v), [], 0.0
    for _ in range(4):
        m.append(np.rint(rest * 128.0))
        rest = rest * 128.0 - m[-1]
    for i in range(4):
        for j in range(4 - i):
            ref = ref + (m[i].T @ m[j]) * 2.0 ** (-7 * (i + j + 2))
    err = (-t2 * D).transpose(0, 2, 1, 3).reshape(o * v, o * v) - ref
    bar = max(1.0, naux / 128.0) * 56 * 2.0 ** -35
    assert abs(float(np.diagonal(err).mean())) <= bar
    assert float(np.abs(err).max()) <= 2.0 * bar
