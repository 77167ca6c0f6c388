"""Performance cases: the work a user of the library has it do, through its
public entry points, over the range of sizes, precisions and directions it is
used at.

listed() names the cases, draw(rng) makes more of the same ranges, prepare()
builds what a program has in hand before the call (inputs, plans, workspaces,
captured graphs), run() is one pass, work() the bytes and flops a pass cannot
do without, exact() the same outputs from plain torch in float64.

Sizes are the benchmark's and the tests': chains of 20 and 100 sites, bonds
32 to 1024, the 784-pixel classifier at batch 4096, the seeded random
tensordot specs (ranks 3-5, dims 8-64), the two-site node split.
"""
from __future__ import annotations

import functools
import math

import torch

from paper_1905_01330_gb300 import synth, tn

LABELS = 10
CHECKPOINT = 28                                  # classifier training: vectors kept every 28 sites
ODD_DIMS = (7, 9, 13, 17, 24, 33, 40, 51)        # leg dimensions off every tile and vector width
SPEC_DIMS = synth.SPEC_DIMS


def listed():
    return [
        # the smallest call: the norm of a short chain, as every normalisation and overlap check asks it
        {"name": "norm_fp32_n20_chi32", "kind": "norm", "n": 20, "chi": 32, "prec": "fp32"},
        # a small network written as ncon labels and planned once: many tiny contractions, launch after launch
        {"name": "ncon_fp32_n20_chi32", "kind": "ncon", "n": 20, "chi": 32, "prec": "fp32"},
        # one contraction of two nodes over two permuted legs, ragged against every tile size
        {"name": "contract_bf16x3_ragged", "kind": "contract", "a": "40,33,56,30", "la": "1,3", "b": "30,48,33,45",
         "lb": "2,0", "prec": "bf16x3"},
        # the benchmark's workload: 2048 uneven contractions as one planned group (the largest case)
        {"name": "group_bf16_2048", "kind": "group", "specs": 2048, "odd": False, "prec": "bf16", "shapes": 2},
        # a group in full float32 precision
        {"name": "group_fp32_256", "kind": "group", "specs": 256, "odd": False, "prec": "fp32", "shapes": 2},
        # energies of one state: a mid-size chain in split bf16, a larger one in float32
        {"name": "energy_bf16x3_n100_chi256", "kind": "energy", "n": 100, "chi": 256, "prec": "bf16x3"},
        {"name": "energy_fp32_n100_chi512", "kind": "energy", "n": 100, "chi": 512, "prec": "fp32"},
        # energies of a batch of states with uneven bonds, planned once and evaluated many times
        {"name": "energy_batch16_bf16x3", "kind": "energy_batch", "n": 100, "states": 16, "lo": 64, "hi": 512,
         "prec": "bf16x3"},
        # classifier inference as a server runs it: the pass captured once, replayed on each new batch
        {"name": "classify_bf16x3_chi128", "kind": "classify", "sites": 784, "chi": 128, "batch": 4096,
         "prec": "bf16x3"},
        # training steps (forward, loss, core gradients): split bf16, and plain float32
        {"name": "train_bf16x3_chi64", "kind": "train", "sites": 784, "chi": 64, "batch": 4096, "prec": "bf16x3"},
        {"name": "train_fp32_chi64", "kind": "train", "sites": 784, "chi": 64, "batch": 4096, "prec": "fp32"},
        # the split of a two-site tensor between its sites, as a sweep does after every update
        {"name": "split_two_site_chi128", "kind": "split", "chi": 128, "keep": 128},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["norm", "ncon", "contract", "group", "energy", "energy_batch", "classify", "train", "split"])
    if kind == "norm":
        return {"kind": kind, "n": _log(rng, 6, 200), "chi": _log(rng, 3, 256),
                "prec": rng.choice(["fp32", "fp32", "bf16x3"])}
    if kind == "ncon":
        return {"kind": kind, "n": _log(rng, 4, 40), "chi": _log(rng, 3, 64), "prec": "fp32"}
    if kind == "contract":
        dims = [_log(rng, 3, 64) for _ in range(6)]   # m0 m1 n0 n1 k0 k1
        m0, m1, n0, n1, k0, k1 = dims
        a = rng.choice([((m0, k0, m1, k1), (1, 3)), ((k1, m0, m1, k0), (3, 0)), ((m0, m1, k0, k1), (2, 3))])
        b = rng.choice([((k0, k1, n0, n1), (0, 1)), ((n0, k1, n1, k0), (3, 1)), ((k1, n0, k0, n1), (2, 0))])
        text = lambda t: ",".join(str(x) for x in t)  # noqa: E731
        return {"kind": kind, "a": text(a[0]), "la": text(a[1]), "b": text(b[0]), "lb": text(b[1]),
                "prec": rng.choice(["fp32", "bf16", "bf16x3"])}
    if kind == "group":
        prec = rng.choice(["bf16", "bf16x3", "fp32"])
        most = {"bf16": 1024, "bf16x3": 512, "fp32": 192}[prec]
        return {"kind": kind, "specs": _log(rng, 4, most), "odd": rng.random() < 0.5, "prec": prec,
                "shapes": rng.randrange(1, 1000)}
    if kind == "energy":
        prec = rng.choice(["bf16", "bf16x3", "fp32"])
        return {"kind": kind, "n": _log(rng, 12, 100), "chi": _log(rng, 12, 512 if prec == "fp32" else 1024),
                "prec": prec}
    if kind == "energy_batch":
        lo = _log(rng, 16, 128)
        return {"kind": kind, "n": _log(rng, 12, 100), "states": _log(rng, 2, 24), "lo": lo,
                "hi": lo + 32 * rng.randrange(1, 9), "prec": rng.choice(["bf16", "bf16x3", "fp32"])}
    if kind == "classify":
        return {"kind": kind, "sites": rng.choice([64, 196, 400, 784]), "chi": _log(rng, 6, 128),
                "batch": _log(rng, 1, 4096), "prec": rng.choice(["bf16", "bf16x3", "fp32"])}
    if kind == "train":
        return {"kind": kind, "sites": rng.choice([64, 196, 400, 784]), "chi": _log(rng, 6, 64),
                "batch": _log(rng, 16, 4096), "prec": rng.choice(["bf16", "bf16x3", "fp32"])}
    chi = _log(rng, 6, 160)
    return {"kind": kind, "chi": chi, "keep": rng.randint(1, 2 * chi)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _chain(n, chi, g, d=2):
    """MPS cores near a product state: a random matrix times one spin direction
    plus noise, N(0, 1/chi) -- a state with an energy well away from zero."""
    bonds = synth.mps_bonds(n, d, chi)
    up = torch.tensor([0.92, 0.39], device="cuda")
    cores = []
    for i in range(n):
        a, b = bonds[i], bonds[i + 1]
        m = torch.randn(a, 1, b, device="cuda", generator=g)
        e = torch.randn(a, d, b, device="cuda", generator=g)
        cores.append(((m * up.view(1, d, 1) + 0.3 * e) / math.sqrt(chi)).contiguous())
    return cores


def _mpo(n):
    return [torch.from_numpy(w).cuda() for w in synth.tfim_mpo(n)]


def _chis(case):
    lo, hi = case["lo"], case["hi"]
    return synth.uneven_chis(case["states"], seed=50, lo=lo, hi=hi, step=32)


def _classifier_cores(case, g):
    """Cores near the identity, delta + N(0, 0.1^2), the label core in the middle."""
    n, chi, ls = case["sites"], case["chi"], case["sites"] // 2
    bonds = [1] + [chi] * (n - 1) + [1]
    cores = []
    for i in range(n):
        a, b = bonds[i], bonds[i + 1]
        shape = (a, 2, LABELS, b) if i == ls else (a, 2, b)
        core = 0.1 * torch.randn(shape, device="cuda", generator=g)
        core += torch.eye(a, b, device="cuda").view((a, 1, 1, b) if i == ls else (a, 1, b))
        cores.append(core.contiguous())
    return cores, ls


def _norm_network(n):
    """<psi|psi> as ncon labels: bra and ket cores, physical legs joined, ends joined."""
    return [(base + i if i > 0 else 0, 100 + i, base + i + 1 if i < n - 1 else 1)
            for base in (1000, 2000) for i in range(n)]


@functools.lru_cache(maxsize=None)
def _specs(count, odd, shapes):
    return tuple(synth.contraction_specs(count, seed=shapes, dims=ODD_DIMS if odd else SPEC_DIMS))


def _spec_list(case):
    return _specs(case["specs"], case["odd"], case["shapes"])


def _out_shape(spec):
    sa, la, sb, lb = spec
    return tuple(sa[p] for p in range(len(sa)) if p not in la) + tuple(sb[p] for p in range(len(sb)) if p not in lb)


def _offsets(sizes):
    """Where each tensor starts in one buffer, on 256-byte boundaries, and the buffer's length."""
    offs, n = [], 0
    for s in sizes:
        offs.append(n)
        n += (s + 63) // 64 * 64
    return offs, n


def _group_tensors(case, seed):
    specs = _spec_list(case)
    in_shapes = [sh for sa, _, sb, _ in specs for sh in (sa, sb)]
    out_shapes = [_out_shape(sp) for sp in specs]
    in_off, n_in = _offsets([math.prod(s) for s in in_shapes])
    out_off, n_out = _offsets([math.prod(s) for s in out_shapes])
    src = torch.randn(n_in, device="cuda", generator=_gen(seed))
    views = [src[o:o + math.prod(s)].view(s) for o, s in zip(in_off, in_shapes)]
    return specs, views, out_shapes, out_off, n_out


def _ints(text):
    return [int(x) for x in text.split(",")]


def _contract_inputs(case, seed):
    g = _gen(seed)
    a = torch.randn(_ints(case["a"]), device="cuda", generator=g)
    b = torch.randn(_ints(case["b"]), device="cuda", generator=g)
    return a, _ints(case["la"]), b, _ints(case["lb"])


def _node(case, seed):
    """A two-site tensor with a spectrum that decays by two orders of magnitude."""
    g, chi = _gen(seed), case["chi"]
    n = 2 * chi
    q1, _ = torch.linalg.qr(torch.randn(n, n, device="cuda", dtype=torch.float64, generator=g))
    q2, _ = torch.linalg.qr(torch.randn(n, n, device="cuda", dtype=torch.float64, generator=g))
    s = torch.logspace(0, -2, n, device="cuda", dtype=torch.float64)
    return ((q1 * s) @ q2).float().view(chi, 2, 2, chi).contiguous()


def _pixels(case, g):
    return torch.rand(case["batch"], case["sites"], device="cuda", generator=g)


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind in ("norm", "energy", "ncon"):
        st["psi"] = _chain(case["n"], case["chi"], _gen(seed))
        if kind == "energy":
            st["mpo"] = _mpo(case["n"])
        if kind == "ncon":
            st["plan"] = tn.NconPlan(st["psi"] + st["psi"], _norm_network(case["n"]), prec=case["prec"])
    elif kind == "contract":
        st["args"] = _contract_inputs(case, seed)
    elif kind == "group":
        specs, views, out_shapes, out_off, n_out = _group_tensors(case, seed)
        out = torch.zeros(n_out, device="cuda")
        items = [(views[2 * i], list(la), views[2 * i + 1], list(lb),
                  out[out_off[i]:out_off[i] + math.prod(out_shapes[i])].view(out_shapes[i]))
                 for i, (_, la, _, lb) in enumerate(specs)]
        st["out"] = out
        st["plan"] = tn.GroupPlan(items, prec=case["prec"])
    elif kind == "energy_batch":
        g = _gen(seed)
        st["states"] = [_chain(case["n"], chi, g) for chi in _chis(case)]
        st["mpo"] = _mpo(case["n"])
        st["plan"] = tn.ExpectGroupedPlan(st["states"], st["mpo"], prec=case["prec"])
    elif kind == "classify":
        g = _gen(seed)
        cores, ls = _classifier_cores(case, g)
        st["new_pixels"] = _pixels(case, g)
        st["pixels"] = st["new_pixels"].clone()
        st["keep"] = (cores, tn.classifier_workspace(cores, ls, LABELS, case["batch"], 0))

        def scores():
            ft, log_scale, _ = tn.mps_classify(cores, ls, st["pixels"], prec=case["prec"], ckpt_every=0,
                                               workspace=st["keep"][1])
            norm = ft.norm(dim=1, keepdim=True)
            return {"ftilde": ft, "log_scale": log_scale, "logits": ft / norm,
                    "log_norm": torch.log(norm[:, 0].double()) + log_scale}

        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            scores()
        torch.cuda.current_stream().wait_stream(side)
        torch.cuda.synchronize()
        st["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(st["graph"]):
            st["scores"] = scores()
    elif kind == "train":
        g = _gen(seed)
        st["cores"], st["ls"] = _classifier_cores(case, g)
        st["pixels"] = _pixels(case, g)
        st["labels"] = torch.randint(0, LABELS, (case["batch"],), device="cuda", generator=g)
        st["ws"] = tn.classifier_workspace(st["cores"], st["ls"], LABELS, case["batch"], CHECKPOINT)
        # the optimiser's gradient buffer, all cores behind one another
        st["flat"] = torch.zeros(sum(c.numel() for c in st["cores"]), device="cuda")
        st["views"] = [v.view_as(c) for v, c in zip(st["flat"].split([c.numel() for c in st["cores"]]), st["cores"])]
    elif kind == "split":
        st["node"] = _node(case, seed)
    else:
        raise ValueError("unknown kind " + kind)
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _energies(r):
    """Energy per normalised state and log <psi|psi> from {e, log, n, log} (last axis)."""
    return {"result": r, "energy": r[..., 0] / r[..., 2] * torch.exp(r[..., 1] - r[..., 3]),
            "log_norm": torch.log(r[..., 2]) + r[..., 3]}


def run(st):
    case = st["case"]
    kind, prec = case["kind"], case.get("prec")
    if kind == "norm":
        return tn.mps_inner(st["psi"], st["psi"], prec=prec)
    if kind == "ncon":
        return st["plan"].run()
    if kind == "contract":
        return tn.contract(*st["args"], prec=prec)
    if kind == "group":
        st["plan"].run()
        return st["out"]
    if kind == "energy":
        return _energies(tn.mps_expect(st["psi"], st["mpo"], prec=prec))
    if kind == "energy_batch":
        return _energies(st["plan"].run())
    if kind == "classify":
        st["pixels"].copy_(st["new_pixels"])
        st["graph"].replay()
        return st["scores"]
    if kind == "train":
        cores, ls, px, ws = st["cores"], st["ls"], st["pixels"], st["ws"]
        ft, log_scale, _ = tn.mps_classify(cores, ls, px, prec=prec, ckpt_every=CHECKPOINT, workspace=ws)
        loss, dft = tn.mps_classify_loss(ft, st["labels"])
        grads = tn.mps_classify_backward(cores, ls, px, dft, ws, prec=prec, ckpt_every=CHECKPOINT)
        torch._foreach_copy_(st["views"], grads)
        return {"loss": loss, "ftilde": ft, "log_scale": log_scale, "grad": st["flat"]}
    # split: singular vectors are defined up to their signs, so the two nodes
    # are handed on as the truncated two-site tensor they stand for
    u, s, vh, dropped = tn.split_node(st["node"], [0, 1], [2, 3], max_singular_values=case["keep"], full_svd=True)
    return {"theta": tn.contract(u * s, [2], vh, [0], prec="fp32"), "s": s, "dropped": dropped}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _chain_work(n, chi, w):
    """(elements of the cores, flops of a sweep with w MPO channels between them; w = None: a norm)."""
    bonds = synth.mps_bonds(n, 2, chi)
    elems = sum(2 * bonds[i] * bonds[i + 1] for i in range(n))
    flops = 0.0
    for i in range(n):
        a, b = bonds[i], bonds[i + 1]
        flops += 4.0 * a * a * b + 4.0 * a * b * b                                # <psi|psi>
        if w is not None:
            wa, wb = w[i], w[i + 1]
            flops += 4.0 * wa * a * a * b + 8.0 * wa * wb * a * b + 4.0 * wb * a * b * b
    return elems, flops


def work(case):
    kind = case["kind"]
    if kind in ("norm", "ncon"):
        elems, flops = _chain_work(case["n"], case["chi"], None)
        return {"bytes": 4.0 * elems, "flops": flops}
    if kind in ("energy", "energy_batch"):
        w = [1] + [3] * (case["n"] - 1) + [1]
        chis = [case["chi"]] if kind == "energy" else _chis(case)
        parts = [_chain_work(case["n"], c, w) for c in chis]
        return {"bytes": 4.0 * sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    if kind in ("contract", "group"):
        specs = _spec_list(case) if kind == "group" else [tuple(_ints(case[k]) for k in ("a", "la", "b", "lb"))]
        sizes = [synth.spec_sizes(sp) for sp in specs]
        return {"bytes": 4.0 * sum(m * k + k * n + m * n for m, n, k in sizes),
                "flops": 2.0 * sum(m * n * k for m, n, k in sizes)}
    if kind in ("classify", "train"):
        n, chi, batch = case["sites"], case["chi"], case["batch"]
        bonds = [1] + [chi] * (n - 1) + [1]
        pairs = [bonds[i] * bonds[i + 1] * (LABELS if i == n // 2 else 1) for i in range(n)]
        elems, passes = 2.0 * sum(pairs), 1 if kind == "classify" else 3    # forward, adjoint, gradient
        return {"bytes": 4.0 * (elems * (1 if kind == "classify" else 2) + batch * (n + LABELS)),
                "flops": 4.0 * batch * sum(pairs) * passes}
    n, keep = 2 * case["chi"], case["keep"]
    return {"bytes": 4.0 * (2 * n * n + n), "flops": 21.0 * n ** 3 + 2.0 * n * n * keep}


# ---------------------------------------------------------------------------
# the same in float64
# ---------------------------------------------------------------------------

def _exact_sweep(cores, mpo):
    """{e, n, log-scale} of a chain by the left environment sweep in float64."""
    n = len(cores)
    env = torch.ones(1, 1, 1, dtype=torch.float64, device="cuda")      # w a a'
    norm = torch.ones(1, 1, dtype=torch.float64, device="cuda")
    le = ln = 0.0
    for i in range(n):
        a = cores[i].double()
        da, d, db = a.shape
        t = (norm @ a.reshape(da, d * db)).reshape(da * d, db)           # bra a, s, ket b'
        norm = a.reshape(da * d, db).t() @ t
        s = norm.abs().max()
        norm, ln = norm / s, ln + torch.log(s)
        if mpo is not None:
            w = mpo[i].double()
            t = torch.einsum("wpq,psb->wqsb", env, a)                    # p bra, q ket
            t = torch.einsum("wxst,wqsb->xbqt", w, t)
            env = (t.reshape(-1, da * d) @ a.reshape(da * d, db)).reshape(w.shape[1], db, db)
            s = env.abs().max()
            env, le = env / s, le + torch.log(s)
    return env.reshape(-1)[0], le, norm.reshape(-1)[0], ln


def _exact_energy(cores, mpo):
    e, le, v, lv = _exact_sweep(cores, mpo)
    return e / v * torch.exp(le - lv), torch.log(v) + lv


def _phi(px, site):
    x = px[:, site].double() * (math.pi / 2)
    return torch.cos(x), torch.sin(x)


def _exact_scores(cores, ls, px):
    """(scores up to a scale, its log) in float64; the scales carry no gradient."""
    batch = px.shape[0]
    half, logs = [], torch.zeros(batch, dtype=torch.float64, device="cuda")
    for sites, left in ((range(ls), True), (range(len(cores) - 1, ls, -1), False)):
        v = torch.ones(batch, 1, dtype=torch.float64, device="cuda")
        for i in sites:
            c = cores[i]
            c0, s0 = _phi(px, i)
            m0, m1 = (c[:, 0], c[:, 1]) if left else (c[:, 0].t(), c[:, 1].t())
            v = c0[:, None] * (v @ m0) + s0[:, None] * (v @ m1)
            m = v.detach().abs().amax(dim=1)
            logs = logs + torch.log(m)
            v = v / m[:, None]
        half.append(v)
    c0, s0 = _phi(px, ls)
    lab = cores[ls]
    f = 0.0
    for ph, s in ((c0, 0), (s0, 1)):
        t = torch.einsum("bc,alc->bal", half[1], lab[:, s])
        f = f + ph[:, None] * torch.einsum("ba,bal->bl", half[0], t)
    return f, logs


def exact(case, seed):
    kind = case["kind"]
    if kind == "norm":
        _, _, v, lv = _exact_sweep(_chain(case["n"], case["chi"], _gen(seed)), None)
        return torch.stack([torch.sign(v), torch.log(v.abs()) + lv])
    if kind == "ncon":
        _, _, v, lv = _exact_sweep(_chain(case["n"], case["chi"], _gen(seed)), None)
        return v * torch.exp(lv)
    if kind == "contract":
        a, la, b, lb = _contract_inputs(case, seed)
        return torch.tensordot(a.double(), b.double(), dims=(la, lb))
    if kind == "group":
        specs, views, out_shapes, out_off, n_out = _group_tensors(case, seed)
        out = torch.zeros(n_out, dtype=torch.float64, device="cuda")
        for i, (_, la, _, lb) in enumerate(specs):
            r = torch.tensordot(views[2 * i].double(), views[2 * i + 1].double(), dims=(list(la), list(lb)))
            out[out_off[i]:out_off[i] + r.numel()] = r.reshape(-1)
        return out
    if kind == "energy":
        e, ln = _exact_energy(_chain(case["n"], case["chi"], _gen(seed)), _mpo(case["n"]))
        return {"result": None, "energy": e, "log_norm": ln}
    if kind == "energy_batch":
        g, mpo = _gen(seed), _mpo(case["n"])
        rows = [_exact_energy(_chain(case["n"], chi, g), mpo) for chi in _chis(case)]
        return {"result": None, "energy": torch.stack([r[0] for r in rows]),
                "log_norm": torch.stack([r[1] for r in rows])}
    if kind == "classify":
        g = _gen(seed)
        cores, ls = _classifier_cores(case, g)
        f, logs = _exact_scores([c.double() for c in cores], ls, _pixels(case, g))
        norm = f.norm(dim=1)
        # one bf16 rounding per site walks over the sites: the logits of a bf16 sweep have no digits to compare
        logits = None if case["prec"] == "bf16" else f / norm[:, None]
        return {"ftilde": None, "log_scale": None, "logits": logits, "log_norm": torch.log(norm) + logs}
    if kind == "train":
        g = _gen(seed)
        cores, ls = _classifier_cores(case, g)
        px = _pixels(case, g)
        y = torch.randint(0, LABELS, (case["batch"],), device="cuda", generator=g)
        params = [c.double().requires_grad_() for c in cores]
        f, _ = _exact_scores(params, ls, px)
        loss = torch.nn.functional.cross_entropy(f / f.norm(dim=1, keepdim=True), y)
        grads = torch.autograd.grad(loss, params)
        grad = None if case["prec"] == "bf16" else torch.cat([x.reshape(-1) for x in grads])
        return {"loss": loss.detach(), "ftilde": None, "log_scale": None, "grad": grad}
    node, keep, n = _node(case, seed).double(), case["keep"], 2 * case["chi"]
    u, s, vh = torch.linalg.svd(node.reshape(n, n))
    theta = (u[:, :keep] * s[:keep]) @ vh[:keep]
    return {"theta": theta.reshape(node.shape), "s": s[:keep], "dropped": s[keep:]}
