"""The work that users of this library have it do, as measurable cases.

Every case is one call of a public entry point on synthetic density-fitted
clusters: (pq|rs) = sum_P B[P,p,q] B[P,r,s] with B[P,p,q] ~ N(0,1) 0.05
exp(-|p-q|/10) symmetrised in (p,q), orbital energies drawn from [-1.5,-0.4]
and [0.2,4.0] Ha, t1 ~ N(0,1) 1e-3 and MP2 amplitudes for t2: the recipe of
the benchmark and the tests.  The kinds are

  energy  t_energy of one cluster           batch  t_energy_batched
  shard   t_energy_triples of a range       df     t_energy_df (ovvv from the DF factors)
  grad    t_energy_vjp / _vjp_triples       frag   t_energy_frag (a fragment projector)
  mp2     mp2_bno_batched

each with the precision that the call is made with: "ozaki" (exact slices, the
mode that meets 1e-7 Ha) or "fp64" (the default of the interface).
"""
import math

import torch

import paper_2412_18553_gb300 as te

EXACT_FLOPS = 1.0e13  # float64 flops that exact() spends at most: about ten seconds


def listed():
    return [
        # a fragment's smallest cluster: a dozen short launches, latency counts
        dict(name="energy_o4v24", kind="energy", nocc=4, nvir=24, precision="ozaki"),
        # the interface's default precision on a small cluster
        dict(name="energy_fp64_o8v40", kind="energy", nocc=8, nvir=40, precision="fp64"),
        # an ordinary embedded cluster
        dict(name="energy_o16v120", kind="energy", nocc=16, nvir=120, precision="ozaki"),
        # an odd number of virtuals: a member size of the uneven cluster batch
        dict(name="energy_o14v145", kind="energy", nocc=14, nvir=145, precision="ozaki"),
        # a large cluster, whole
        dict(name="energy_o24v240", kind="energy", nocc=24, nvir=240, precision="ozaki"),
        # one shard of the benchmark's cluster: a user spreads its 5952 triples over calls
        dict(name="shard_o32v320", kind="shard", nocc=32, nvir=320, first=2976, count=48, precision="ozaki"),
        # the clusters of one molecule in one call, sizes uneven
        dict(name="batch_6", kind="batch", members=6, omin=8, omax=14, precision="ozaki"),
        # the gradient of an ordinary cluster, all seven inputs
        dict(name="grad_o16v120", kind="grad", nocc=16, nvir=120, first=0, count=0, precision="ozaki"),
        # a range of a large cluster's gradient (five slices per element)
        dict(name="grad_o8v320", kind="grad", nocc=8, nvir=320, first=60, count=4, precision="ozaki"),
        # the fragment-projected energy of an ordinary cluster
        dict(name="frag_o16v120", kind="frag", nocc=16, nvir=120, rank=6, precision="ozaki"),
        # the energy of a cluster that is given by its density-fitting factors
        dict(name="df_o16v160", kind="df", nocc=16, nvir=160, naux=704, precision="ozaki"),
        # the step before the triples for a batch of clusters: amplitudes, densities, populations
        dict(name="mp2_8", kind="mp2", members=8, omin=8, omax=20, precision="fp64"),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    while True:
        kind = rng.choice(("energy", "energy", "shard", "batch", "df", "grad", "grad", "frag", "mp2"))
        precision = "fp64" if kind in ("energy", "grad", "frag", "mp2") and rng.random() < 0.25 else "ozaki"
        if kind in ("energy", "grad", "frag"):
            # whole clusters (the float64 ones smaller: their rate is a hundredth)
            top_o, top_v = (24, 240) if kind == "energy" else (16, 120)
            if precision == "fp64":
                top_o, top_v = (14, 96) if kind == "energy" else (8, 48)
            case = dict(kind=kind, nocc=_log(rng, 3, top_o), nvir=_log(rng, 12, top_v), precision=precision)
            if kind == "frag":
                case["rank"] = rng.randint(1, case["nocc"] - 1)
            if kind == "grad":
                case.update(first=0, count=0)
                if precision == "ozaki" and rng.random() < 0.5:  # a range of a larger cluster
                    case.update(nocc=rng.randint(3, 10), nvir=rng.randint(121, 320))
                    case["first"] = rng.randrange(te.num_unique_triples(case["nocc"]) - 6)
                    case["count"] = rng.randint(1, 6)
        elif kind == "shard":
            case = dict(kind=kind, nocc=_log(rng, 4, 32), nvir=_log(rng, 120, 560), precision=precision)
            nt = te.num_unique_triples(case["nocc"])
            case["count"] = min(nt, _log(rng, 4, 64))
            case["first"] = rng.randint(0, nt - case["count"])
        elif kind == "df":
            case = dict(kind=kind, nocc=_log(rng, 3, 20), nvir=_log(rng, 16, 200), precision=precision)
            case["naux"] = int(rng.uniform(2.0, 4.0) * (case["nocc"] + case["nvir"]))
        else:
            case = dict(kind=kind, members=rng.randint(2, 8 if kind == "batch" else 12), precision=precision)
            case["omin"] = rng.randint(4, 10)
            case["omax"] = case["omin"] + rng.randint(0, 6 if kind == "batch" else 10)
        bytes_ = max(8.0 * o * v ** 3 for o, v in _sizes(case)) if kind != "mp2" else 0.0
        if bytes_ <= 9e9 and work(case)["flops"] <= 5e13:
            return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _sizes(case):
    """(nocc, nvir) of every cluster of a case; batches: nvir about 8 nocc, odd and even."""
    if "members" not in case:
        return [(case["nocc"], case["nvir"])]
    n, lo, hi = case["members"], case["omin"], case["omax"]
    occ = [lo + (hi - lo) * k // max(1, n - 1) for k in range(n)]
    return [(o, 8 * o + (k % 3) - 1) for k, o in enumerate(occ)]


def _factor(o, v, naux, gen, dev):
    n = o + v
    idx = torch.arange(n, dtype=torch.float64, device=dev)
    env = 0.05 * torch.exp(-(idx[:, None] - idx[None, :]).abs() / 10.0)
    B = torch.randn((naux, n, n), dtype=torch.float64, device=dev, generator=gen) * env
    B = 0.5 * (B + B.transpose(1, 2))
    eps_o = (torch.rand(o, dtype=torch.float64, device=dev, generator=gen) * 1.1 - 1.5).sort().values
    eps_v = (torch.rand(v, dtype=torch.float64, device=dev, generator=gen) * 3.8 + 0.2).sort().values
    t1 = torch.randn((o, v), dtype=torch.float64, device=dev, generator=gen) * 1e-3
    return eps_o, eps_v, B, t1


def _ovvv(Bov, Bvv):
    """sum_P Bov[P,i,a] Bvv[P,b,d]: float64 where that is quick, else from
    float32 parts (all bits of the sum are kept; the arrays are the inputs)."""
    P, o, v = Bov.shape
    lhs, rhs = Bov.reshape(P, o * v).T, Bvv.reshape(P, v * v)
    if 2.0 * o * v ** 3 * P <= 2e11:
        return (lhs @ rhs).reshape(o, v, v, v)
    lh, rh = lhs.float(), rhs.float()
    ll, rl = (lhs - lh.double()).float(), (rhs - rh.double()).float()
    out = torch.empty((o, v, v, v), dtype=torch.float64, device=Bov.device)
    for i in range(o):  # an occupied index at a time: no second array of ovvv's size
        s = slice(i * v, (i + 1) * v)
        out[i] = (lh[s] @ rh).double().add_((lh[s] @ rl).add_(ll[s] @ rh)).reshape(v, v, v)
    return out


def _cluster(o, v, naux, gen, dev, with_df=False):
    eps_o, eps_v, B, t1 = _factor(o, v, naux, gen, dev)
    Boo, Bov, Bvv = (B[:, :o, :o].contiguous(), B[:, :o, o:].contiguous(), B[:, o:, o:].contiguous())
    ov = Bov.reshape(naux, o * v)
    ovov = (ov.T @ ov).reshape(o, v, o, v)
    ooov = (Boo.reshape(naux, o * o).T @ ov).reshape(o, o, o, v)
    d2 = (eps_o[:, None, None, None] + eps_o[None, :, None, None]
          - eps_v[None, None, :, None] - eps_v[None, None, None, :])
    t2 = (ovov.permute(0, 2, 1, 3) / d2).contiguous()
    c = dict(eps_o=eps_o, eps_v=eps_v, ooov=ooov, ovov=ovov, t1=t1, t2=t2)
    if with_df:
        return c, Bov, Bvv
    c["ovvv"] = _ovvv(Bov, Bvv)
    return c


def _inputs(case, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    kind, sizes = case["kind"], _sizes(case)
    if kind == "mp2":
        out = []
        for o, v in sizes:
            eps_o, eps_v, B, _ = _factor(o, v, 4 * (o + v), gen, dev)
            out.append((eps_o, eps_v, B[:, :o, o:].contiguous()))
        return out
    if kind == "batch":
        return [_cluster(o, v, 4 * (o + v), gen, dev) for o, v in sizes]
    o, v = sizes[0]
    if kind == "df":
        return _cluster(o, v, case["naux"], gen, dev, with_df=True)
    c = _cluster(o, v, 4 * (o + v), gen, dev)
    if kind == "frag":  # the projector onto a fragment: rank orthonormal columns
        q, _ = torch.linalg.qr(torch.randn((o, o), dtype=torch.float64, device=dev, generator=gen))
        return c, (q[:, :case["rank"]] @ q[:, :case["rank"]].T).contiguous()
    return c


def prepare(case, seed):
    """The cluster's arrays on the GPU.  The library's default handle keeps its
    workspace between calls, as in a user's program."""
    return dict(case, data=_inputs(case, seed))


def run(state):
    kind, data, p = state["kind"], state["data"], state["precision"]
    if kind == "energy":
        return te.t_energy(data, p)
    if kind == "shard":
        return te.t_energy_triples(data, state["first"], state["first"] + state["count"], p)
    if kind == "batch":
        return te.t_energy_batched(data, p)
    if kind == "df":
        return te.t_energy_df(*data, p)
    if kind == "frag":
        return te.t_energy_frag(data[0], data[1], p, shares=True)
    if kind == "grad":
        if state["count"]:
            return te.t_energy_vjp_triples(data, state["first"], state["first"] + state["count"], precision=p)
        return te.t_energy_vjp(data, precision=p)
    return te.mp2_bno_batched(data, p)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    """Flops of the contractions, 12 v^3 (v + o) per occupied triple (three
    times that for the gradient and the projected energy); the inputs read and
    the outputs written once."""
    kind, flops, nbytes = case["kind"], 0.0, 0.0
    for o, v in _sizes(case):
        nt = te.num_unique_triples(o)
        small = 8.0 * (o ** 3 * v + 2.0 * o * o * v * v + o * v + o + v)  # ooov, ovov, t2, t1, eps
        per = 12.0 * float(v) ** 3 * (v + o)
        if kind == "mp2":
            P = 4 * (o + v)
            flops += te.mp2_flop_count(o, v, P)
            nbytes += 8.0 * (P * o * v + o + v + o * o * v * v + o * o + v * v + o + v)
        elif kind == "df":
            P = case["naux"]
            flops += nt * per + 2.0 * o * float(v) ** 3 * P
            nbytes += small + 8.0 * P * (o * v + v * v)
        elif kind == "grad":
            flops += 3.0 * (case["count"] or nt) * per
            nbytes += 2.0 * (small + 8.0 * o * float(v) ** 3)
        elif kind == "shard":
            flops += case["count"] * per
            nbytes += small + 8.0 * o * float(v) ** 3 + 8.0 * case["count"]
        else:
            flops += (3.0 if kind == "frag" else 1.0) * nt * per
            nbytes += small + 8.0 * o * float(v) ** 3 + (8.0 * nt if kind == "frag" else 8.0)
    return dict(bytes=nbytes, flops=flops)


# ---------------------------------------------------------------------------
# the same results in float64 with plain torch
# ---------------------------------------------------------------------------

def _triples(o):
    return [(i, j, k) for i in range(o) for j in range(i + 1) for k in range(j + 1) if not i == j == k]


def _mult(t):
    return 3.0 if len(set(t)) == 2 else 6.0


def _x(c, p, q, r):
    """X_pqr[a,b,c] = sum_d (pa|bd) t_rq^cd - sum_l (pa|ql) t_lr^bc."""
    return torch.einsum("abd,cd->abc", c["ovvv"][p], c["t2"][r, q]) - torch.einsum("la,lbc->abc", c["ooov"][q, :, p], c["t2"][:, r])


# the six terms of P: occupied positions of X, and the order of its indices
# that gives [a, b, c]
_P6 = (((0, 1, 2), (0, 1, 2)), ((1, 2, 0), (2, 0, 1)), ((2, 0, 1), (1, 2, 0)),
       ((0, 2, 1), (0, 2, 1)), ((2, 1, 0), (2, 1, 0)), ((1, 0, 2), (1, 0, 2)))


def _w(c, t):
    return sum(_x(c, *(t[n] for n in occ)).permute(*vir) for occ, vir in _P6)


def _y(c, t):
    one = lambda p, q, r: c["ovov"][p, :, q, :, None] * c["t1"][r]  # noqa: E731
    return 0.5 * sum(one(*(t[n] for n in occ)).permute(*vir) for occ, vir in _P6)


def _d(c, t):
    ev = c["eps_v"]
    return c["eps_o"][list(t)].sum() - ev[:, None, None] - ev[None, :, None] - ev[None, None, :]


def _r(x):
    return (4.0 * x + x.permute(1, 2, 0) + x.permute(2, 0, 1) - 2.0 * (x.permute(2, 1, 0) + x.permute(0, 2, 1) + x.permute(1, 0, 2)))


def _share(c, t):
    w = _w(c, t)
    return _mult(t) / 3.0 * (w * _r(w + _y(c, t)) / _d(c, t)).sum()


def _exact_grad(c, triples):
    """The gradient of the sum of the triples' shares: one reverse step per
    triple, written out."""
    g = {n: torch.zeros_like(x) for n, x in c.items()}
    total, t2, ooov, ovvv = 0.0, c["t2"], c["ooov"], c["ovvv"]
    for t in triples:
        s = _mult(t) / 3.0
        w, y, d = _w(c, t), _y(c, t), _d(c, t)
        rw, rv = _r(w), _r(w + y)
        e = w * rv / d
        total = total + s * e.sum()
        dw, dy, dd = s * (rw + rv) / d, s * rw / d, -s * e / d
        g["eps_o"].index_add_(0, torch.tensor(t, device=dd.device), dd.sum().expand(3))
        g["eps_v"] -= dd.sum((1, 2)) + dd.sum((0, 2)) + dd.sum((0, 1))
        for occ, vir in _P6:
            p, q, r = (t[n] for n in occ)
            inv = [vir.index(n) for n in range(3)]
            dx = dw.permute(*inv).contiguous()  # the gradient of X_pqr[a,b,c]
            du = 0.5 * dy.permute(*inv)
            g["ovvv"][p] += torch.einsum("abc,cd->abd", dx, t2[r, q])
            g["t2"][r, q] += torch.einsum("abc,abd->cd", dx, ovvv[p])
            g["ooov"][q, :, p] -= torch.einsum("abc,lbc->la", dx, t2[:, r])
            g["t2"][:, r] -= torch.einsum("abc,la->lbc", dx, ooov[q, :, p])
            g["ovov"][p, :, q] += torch.einsum("abc,c->ab", du, c["t1"][r])
            g["t1"][r] += torch.einsum("abc,ab->c", du, c["ovov"][p, :, q])
    return total, g


def _exact_frag(c, cf):
    """E_x with W~ projected in each of its occupied indices in turn (a third each)."""
    o = c["eps_o"].shape[0]
    kept = {}

    def w(*t):
        order = sorted(range(3), key=lambda n: -t[n])  # W~ is unchanged when (p,a), (q,b), (r,c) change places
        key = tuple(t[n] for n in order)
        if key not in kept:
            kept[key] = _w(c, key)
        return kept[key].permute(*[order.index(n) for n in range(3)])

    shares = []
    for t in _triples(o):
        sw = torch.zeros_like(w(*t))
        for n in range(3):
            for p in range(o):
                sw += cf[t[n], p] * w(*t[:n], p, *t[n + 1:])
        shares.append(_mult(t) / 9.0 * (sw * _r(w(*t) + _y(c, t)) / _d(c, t)).sum())
    shares = torch.stack(shares)
    return shares.sum(), shares


def _exact_mp2(eps_o, eps_v, B):
    ovov = torch.einsum("Pia,Pjb->ijab", B, B)
    t2 = -ovov / (eps_v[:, None] + eps_v[None, :] - eps_o[:, None, None, None] - eps_o[:, None, None])
    tt = 2.0 * t2 - t2.transpose(2, 3)
    gvv = 2.0 * torch.einsum("ijac,ijbc->ab", t2, tt)
    goo = 2.0 * torch.eye(len(eps_o), dtype=t2.dtype, device=t2.device) - 2.0 * torch.einsum("ikab,jkab->ij", t2, tt)
    pop = lambda g: torch.linalg.eigvalsh(0.5 * (g + g.T))  # noqa: E731
    return dict(t2=t2, gamma_oo=goo, gamma_vv=gvv, pop_o=pop(goo), pop_v=pop(gvv))


def exact(case, seed):
    if work(case)["flops"] > EXACT_FLOPS:
        return None
    kind, data = case["kind"], _inputs(case, seed)
    if kind == "mp2":
        return [_exact_mp2(*c) for c in data]
    if kind == "batch":
        return torch.stack([sum(_share(c, t) for t in _triples(len(c["eps_o"]))) for c in data])
    if kind == "frag":
        return _exact_frag(*data)
    if kind == "df":
        c, Bov, Bvv = data
        P, o, v = Bov.shape
        data = dict(c, ovvv=(Bov.reshape(P, o * v).T @ Bvv.reshape(P, v * v)).reshape(o, v, v, v))
    triples = _triples(len(data["eps_o"]))
    if kind == "shard":
        return torch.stack([_share(data, t) for t in triples[case["first"]:case["first"] + case["count"]]])
    if kind == "grad":
        return _exact_grad(data, triples[case["first"]:case["first"] + case["count"]] if case["count"] else triples)
    return sum(_share(data, t) for t in triples)
