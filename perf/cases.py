"""Workloads of this framework whose speed is measured, with their inputs and exact results.

A case is a dict of plain values; its "kind" names the public call that is measured:

  flow     one sweep of a Quantum Flow through the handle API (`qflow.Flow`) from a given pool, as a
           program that drives a flow (or restarts one from a stored pool) makes it: the pool in, one
           sweep, the mean and per-space energies and the new pool out, all through host buffers.
           The pool is the one two sweeps from the empty pool leave: the middle of a run, which
           takes about six sweeps.
  dress    the dressing alone (`qflow.dress_device`, FP64) on device tensors.
  solve    the solver of one size class (`qflow.solve_device`) on device tensors.
  train    one optimiser step of the warm-start network: gradient and Adam.
  infer    the warm-start network's forward pass.

Systems follow the recipe of the package's synthetic inputs (`synth`); their sizes are the package's
own systems, and draw() spreads sizes, space lists and forms over the ranges between them.
"""
import itertools
import math

import numpy as np
import torch

from paper_2606_04186_gb300 import qflow, synth


def _flow(n, nocc, xi, spaces, count, precision, form="ses"):
    return {"kind": "flow", "n": n, "nocc": nocc, "xi": xi, "spaces": spaces, "count": count, "precision": precision,
            "form": form}


def listed():
    return [
        # the smallest system: 35 spaces, where a sweep is launches and latencies (default precision)
        dict(_flow(10, 3, 3.0, "all", 35, "fp64"), name="n10_all_fp64"),
        # a small molecule, every 6e6o space, in the plain FP64 form and in the mixed form
        dict(_flow(24, 5, 4.0, "all", 9690, "fp64"), name="n24_all_fp64"),
        dict(_flow(24, 5, 4.0, "all", 9690, "mixed"), name="n24_all_mixed"),
        # the same in the Hermitian form of the paper (FP64 only)
        dict(_flow(24, 5, 4.0, "all", 9690, "fp64", "ducc"), name="n24_all_ducc"),
        # 2e2o, 4e4o and 6e6o spaces in one list, 20,000 of each
        dict(_flow(40, 6, 4.0, "mixed", 20000, "mixed"), name="n40_sizes_mixed"),
        # a coverage cycle of Algorithm 1 on 82 orbitals (about 35,600 spaces, cut to a fixed count)
        # in FP64: the paper's way to choose the spaces of a sweep
        dict(_flow(82, 10, 5.0, "cycle", 35000, "fp64"), name="n82_cycle_fp64"),
        # the largest runs: every 6e6o space of 82 orbitals, and 2,000,000 of 114 orbitals
        dict(_flow(82, 10, 5.0, "all", 7156800, "mixed"), name="n82_all_mixed"),
        dict(_flow(114, 11, 8.0, "sample", 2000000, "mixed"), name="n114_sample_mixed"),
        # dressing alone: a mid size with odd dimensions, for programs that own the solver's side
        {"kind": "dress", "n": 57, "nocc": 7, "xi": 5.0, "name": "dress_n57_fp64"},
        # the solver alone on one size class, FP64 (the default) and an odd count
        {"kind": "solve", "n": 40, "nocc": 6, "xi": 4.0, "k": 2, "count": 8191, "precision": "fp64", "name": "solve_4e4o_fp64"},
        # the network: a training step at the batch size its training uses, and inference at the
        # row count of a warm start's chunk
        {"kind": "train", "hidden": 256, "rows": 128, "name": "mlp_train_128"},
        {"kind": "infer", "hidden": 256, "rows": 131072, "name": "mlp_infer_131072"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["flow", "flow", "flow", "flow", "dress", "solve", "train", "infer"])
    if kind == "train":
        return {"kind": kind, "hidden": rng.randint(32, 320), "rows": _log_int(rng, 16, 4096)}
    if kind == "infer":
        return {"kind": kind, "hidden": rng.randint(32, 320), "rows": _log_int(rng, 64, 131072)}
    xi = round(rng.uniform(3.0, 8.0), 2)
    if kind == "dress":
        n = _log_int(rng, 10, 96)
        return {"kind": kind, "n": n, "nocc": rng.randint(3, min(11, n // 2)), "xi": xi}
    if kind == "solve":
        n = rng.randint(16, 60)
        return {"kind": kind, "n": n, "nocc": rng.randint(4, 8), "xi": xi, "k": rng.randint(1, 3),
                "count": _log_int(rng, 50, 50000), "precision": rng.choice(["fp64", "mixed"])}
    form = rng.choice(["mixed", "mixed", "fp64", "fp64", "ducc"])
    if form == "ducc":
        n = rng.randint(10, 32)
        return _flow(n, rng.randint(3, 6), xi, rng.choice(["sample", "mixed"]), _log_int(rng, 35, 5000), "fp64", "ducc")
    n = _log_int(rng, 10, 114 if form == "mixed" else 82)
    nocc = rng.randint(3, min(11, n // 3))
    spaces = rng.choice(["sample", "mixed", "cycle"])
    tuples = math.comb(nocc, 2) * math.comb(n - nocc, 2)  # a cycle has about a third as many spaces
    most = tuples // 3 if spaces == "cycle" else 1000000
    return _flow(n, nocc, xi, spaces, _log_int(rng, min(35, most), min(most, 1000000 if form == "mixed" else 20000)), form)


# ---- inputs --------------------------------------------------------------------------------------


def _space_list(case, eps, seed):
    """The case's list of active spaces (int32 records)."""
    n, no, cnt = case["n"], case["nocc"], case["count"]
    most = math.comb(no, 3) * math.comb(n - no, 3)
    if case["spaces"] == "all":
        return synth.all_spaces(n, no)
    if case["spaces"] == "mixed":
        return synth.mixed_spaces(n, no, min(cnt, most), seed)
    if case["spaces"] == "cycle":  # the first `count` spaces of one coverage cycle after another
        sp = [qflow.sample_spaces(eps, no, 3, 3, seed)[0]]
        while sum(map(len, sp)) < cnt:
            sp.append(qflow.sample_spaces(eps, no, 3, 3, seed + len(sp))[0])
        return np.concatenate(sp)[:cnt]
    return synth.sampled_spaces(n, no, min(cnt, most), seed)


def _system(case, seed):
    return synth.make_system(case["n"], case["nocc"], case["xi"], seed)


def _class_spaces(case, seed):
    n, no, k = case["n"], case["nocc"], case["k"]
    cnt = min(case["count"], math.comb(no, k) * math.comb(n - no, k))
    return synth.sampled_spaces(n, no, cnt, seed, no=k, nv=k)


def _net(case, seed):
    """Parameters, standardised inputs and targets of the network case."""
    rng = np.random.default_rng(seed)
    p = synth.mlp_init_params(qflow.MLP_NIN, case["hidden"], qflow.MLP_NOUT, seed).astype(np.float32)
    x = rng.standard_normal((case["rows"], qflow.MLP_NIN), dtype=np.float32)
    t = rng.standard_normal((case["rows"], qflow.MLP_NOUT), dtype=np.float32)
    return p, x, t


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "flow":
        eps, h, eri = _system(case, seed)
        fl = qflow.Flow(h, eri, case["nocc"], _space_list(case, eps, seed + 1), precision=case["precision"],
                        form=case["form"])
        for _ in range(2):
            fl.sweep(raise_on_fail=False)
        t1, t2 = fl.amplitudes()
        fl.sweep(raise_on_fail=False)  # launch schedule and graph are fixed by the third sweep
        return {"kind": kind, "flow": fl, "t1": t1, "t2": t2}
    if kind in ("dress", "solve"):
        n, no = case["n"], case["nocc"]
        eps, h, eri = _system(case, seed)
        t1, t2 = synth.random_amplitudes(no, n - no, seed, 0.01, 0.02)
        f64 = lambda *s: torch.zeros(s, dtype=torch.float64, device="cuda")  # noqa: E731
        s = {"kind": kind, "n": n, "nocc": no, "h": _cuda(h), "eri": _cuda(eri), "t1": _cuda(t1), "t2": _cuda(t2)}
        if kind == "dress":
            s.update(e0=f64(1), F=f64(n, n), W=f64(n, n, n, n),
                     work=torch.empty(qflow.dress_workspace(n, no), dtype=torch.uint8, device="cuda"))
            return s
        # dressed integrals of the first sweep (empty pool) with a pool of earlier amplitudes
        e0, F, W = _dress64(s["h"], s["eri"], torch.zeros_like(s["t1"]), torch.zeros_like(s["t2"]), no)
        sp = _class_spaces(case, seed + 1)
        perm, o1, o2, _ = qflow.plan(h, eri, no, sp)
        cnt = len(sp)
        s.update(e0=e0.reshape(1), F=F, W=W, k=case["k"], precision=case["precision"], spaces=_cuda(sp[perm]),
                 owner1=_cuda(o1), owner2=_cuda(o2), t1n=f64(*t1.shape), t2n=f64(*t2.shape), energy=f64(cnt),
                 status=torch.zeros(cnt, dtype=torch.int32, device="cuda"))
        return s
    p, x, t = _net(case, seed)
    H, rows = case["hidden"], case["rows"]
    work = torch.empty(qflow.mlp_workspace(qflow.MLP_NIN, H, qflow.MLP_NOUT, rows), dtype=torch.uint8, device="cuda")
    s = {"kind": kind, "hidden": H, "p": _cuda(p), "x": _cuda(x), "work": work}
    if kind == "infer":
        s["y"] = torch.empty((rows, qflow.MLP_NOUT), dtype=torch.float32, device="cuda")
        return s
    s.update(t=_cuda(t), grad=torch.empty_like(s["p"]), loss=torch.empty(1, dtype=torch.float32, device="cuda"),
             p0=s["p"].clone(), m=torch.zeros_like(s["p"]), v=torch.zeros_like(s["p"]))
    return s


# ---- one pass ------------------------------------------------------------------------------------


def run(s):
    kind = s["kind"]
    stream = torch.cuda.current_stream().cuda_stream
    if kind == "flow":
        fl = s["flow"]
        fl.set_amplitudes(s["t1"], s["t2"])
        nfailed = fl.sweep(raise_on_fail=False)[2]
        mean, energies = fl.energy(per_space=True)
        t1, t2 = fl.amplitudes()
        return {"mean": mean, "energies": energies, "nfailed": nfailed, "t1": t1, "t2": t2}
    if kind == "dress":
        qflow.dress_device(s["h"], s["eri"], s["t1"], s["t2"], s["nocc"], s["e0"], s["F"], s["W"], s["work"], stream)
        return {"e0": s["e0"], "F": s["F"], "W": s["W"]}
    if kind == "solve":
        s["t1n"].copy_(s["t1"])
        s["t2n"].copy_(s["t2"])
        qflow.solve_device(s["n"], s["nocc"], s["e0"], s["F"], s["W"], s["k"], s["spaces"], s["energy"], s["status"],
                           owner1=s["owner1"], owner2=s["owner2"], t1_old=s["t1"], t2_old=s["t2"], t1_new=s["t1n"],
                           t2_new=s["t2n"], precision=s["precision"], stream=stream)
        return {"energy": s["energy"], "status": s["status"], "t1": s["t1n"], "t2": s["t2n"]}
    nin, nout, H = qflow.MLP_NIN, qflow.MLP_NOUT, s["hidden"]
    if kind == "infer":
        qflow.mlp_forward_device(nin, H, nout, s["p"], s["x"], s["y"], s["work"], stream)
        return {"y": s["y"]}
    # the step starts from the same parameters and moments at every pass
    s["p"].copy_(s["p0"])
    s["m"].zero_()
    s["v"].zero_()
    qflow.mlp_grad_device(nin, H, nout, s["p"], s["x"], s["t"], s["grad"], s["loss"], s["work"], stream=stream)
    qflow.mlp_adam_device(s["p"], s["grad"], s["m"], s["v"], 1, 2e-3, stream=stream)
    return {"loss": s["loss"], "grad": s["grad"], "m": s["m"], "v": s["v"], "params": s["p"]}


# ---- work ----------------------------------------------------------------------------------------


def _dress_flops(n, o):
    """Two operations per term of the dressing's contractions, every element of every block."""
    v = n - o
    t1 = 4 * o * v * n**3
    gemm = (o**4 * v**2 + 4 * (o * v) ** 3 + o * o * v * v * (v * v + o * o) + 10 * (o * v) ** 3 + v**4 * o * o
            + 3 * (o * v) ** 3 + o**3 * v**3 + 3 * o**4 * v**2 + v**3 * o * (3 * o * v + o * o))
    return 2.0 * (t1 + gemm)


def _solve_flops(k, count, precision):
    """Operations of `count` spaces: the determinant operator applied to spin-symmetric vectors, once
    (mixed, where most spaces stop after one step from the first-order vector) or five times (FP64)."""
    ns, nsg = {1: (2, 2), 2: (6, 6), 3: (20, 12)}[k]
    ndet = ns * (ns + 1) // 2
    return count * (1 if precision == "mixed" else 5) * ndet * (2.0 * nsg * nsg + 4 * ns + 2)


def work(case):
    kind = case["kind"]
    if kind in ("train", "infer"):
        H, rows = case["hidden"], case["rows"]
        params = qflow.MLP_NIN * H + H * H + H * qflow.MLP_NOUT
        io = rows * (qflow.MLP_NIN + qflow.MLP_NOUT)
        if kind == "infer":
            return {"bytes": 4.0 * (params + io), "flops": 2.0 * rows * params}
        return {"bytes": 4.0 * (7 * params + io), "flops": 2.0 * rows * (3 * params - qflow.MLP_NIN * H)}
    n, o = case["n"], case["nocc"]
    pool = o * (n - o) + (o * (n - o)) ** 2
    if kind == "dress":
        return {"bytes": 8.0 * (2 * n**4 + pool), "flops": _dress_flops(n, o)}
    if kind == "solve":
        k, cnt = case["k"], min(case["count"], math.comb(o, case["k"]) * math.comb(n - o, case["k"]))
        return {"bytes": 8.0 * (min(n**4, cnt * (2 * k) ** 4) + 2 * pool) + 44.0 * cnt, "flops": _solve_flops(k, cnt, case["precision"])}
    most = math.comb(o, 3) * math.comb(n - o, 3)
    cnt = case["count"] if case["spaces"] == "cycle" else most if case["spaces"] == "all" else min(case["count"], most)
    small = 0.0
    if case["spaces"] == "mixed":
        small = _solve_flops(1, cnt, case["precision"]) + _solve_flops(2, cnt, case["precision"])
    dressings = 8 if case["form"] == "ducc" else 1
    return {"bytes": 8.0 * (n**4 + 2 * pool) + 40.0 * cnt,
            "flops": dressings * _dress_flops(n, o) + _solve_flops(3, cnt, case["precision"]) + small}


# ---- exact results (64 bits, torch and numpy only) -------------------------------------------------


def _dress64(h, g, t1, t2, o):
    """E0, F, W of e^{-T} H e^{T} in normal order, cut after two-body terms."""
    n = h.shape[0]
    K = torch.zeros_like(h)
    K[o:, :o] = t1.T
    X, Y = torch.eye(n, dtype=h.dtype, device=h.device) - K, torch.eye(n, dtype=h.dtype, device=h.device) + K
    ht = X @ h @ Y
    w = X @ g.reshape(n, -1)
    w = (Y.T @ w.reshape(n, n, n * n)).reshape(n * n, n, n)
    w = (X @ w) @ Y
    W = w.reshape(n, n, n, n)
    O, V = slice(0, o), slice(o, n)
    es = torch.einsum
    F = ht + 2 * es("pqkk->pq", W[:, :, O, O]) - es("pkkq->pq", W[:, O, O, :])
    u = 2 * t2 - t2.transpose(2, 3)
    oovv = W[O, V, O, V].permute(0, 2, 1, 3).contiguous()  # [m n e f] = g~_menf
    e0 = 2 * torch.trace(ht[O, O]) + 2 * es("kkll->", W[O, O, O, O]) - es("kllk->", W[O, O, O, O]) + (oovv * u).sum()
    fov = F[O, V]
    foo = F[O, O] + es("mnef,inef->mi", oovv, u)
    fvv = F[V, V] - es("mnef,mnaf->ae", oovv, u)
    r1 = (F[V, O] + es("me,imae->ai", fov, u) + es("aemf,imef->ai", W[V, V, O, V], u) - es("mine,mnae->ai", W[O, O, O, V], u))
    wo = W[O, O, O, O] + es("klef,ijef->kilj", oovv, t2)
    # doubles block
    r2 = W[V, O, V, O].permute(1, 3, 0, 2).clone()  # [i j a b]
    sym = es("be,ijae->ijab", fvv, t2) - es("mj,imab->ijab", foo, t2)
    ovvo, oovv2 = W[O, V, V, O], W[O, O, V, V]
    sym = sym + es("mebj,imae->ijab", ovvo, u) - es("mjbe,imae->ijab", oovv2, t2) - es("mibe,jmea->ijab", oovv2, t2)
    r2 = r2 + sym + sym.permute(1, 0, 3, 2)
    r2 = r2 + es("minj,mnab->ijab", wo, t2) + es("aebf,ijef->ijab", W[V, V, V, V], t2)
    A = es("imae,mnef->ianf", u, oovv)
    B = es("imae,mnfe->ianf", u, oovv)
    C = es("imae,mnfe->ianf", t2, oovv)
    D = es("jmea,mnfe->janf", t2, oovv)
    r2 = r2 + es("ianf,jnbf->ijab", A, u) - es("ianf,jnbf->ijab", B, t2) + es("ianf,jnfb->ijab", C, t2) + es("janf,infb->ijab", D, t2)
    # remaining two-body blocks
    n_ovvo = ovvo + es("mnef,jnbf->mebj", oovv, u) - es("mnfe,jnbf->mebj", oovv, t2)
    n_oovv = oovv2 - es("infb,jnfa->ijab", oovv, t2)
    n_oovo = (W[O, O, V, O] + es("me,ijeb->mibj", fov, t2) + es("mebf,ijef->mibj", W[O, V, V, V], t2)
              + es("mine,jnbe->mibj", W[O, O, O, V], u) - es("meni,jnbe->mibj", W[O, V, O, O], t2) - es("menj,ineb->mibj", W[O, V, O, O], t2))
    n_vvvo = (W[V, V, V, O] - es("me,miab->aebi", fov, t2) + es("meni,mnab->aebi", W[O, V, O, O], t2)
              + es("mfae,mifb->aebi", W[O, V, V, V], u) - es("mebf,miaf->aebi", W[O, V, V, V], t2) - es("meaf,mifb->aebi", W[O, V, V, V], t2))
    n_vvvv = W[V, V, V, V] + es("mnef,mnab->aebf", oovv, t2)
    Wd = W.clone()
    Wd[O, O, O, O] = wo
    Wd[V, O, V, O] = r2.permute(2, 0, 3, 1)
    Wd[V, V, V, V] = n_vvvv
    Wd[O, V, V, O] = n_ovvo
    Wd[V, O, O, V] = n_ovvo.permute(2, 3, 0, 1)
    Wd[O, O, V, V] = n_oovv
    Wd[V, V, O, O] = n_oovv.permute(2, 3, 0, 1)
    Wd[O, O, V, O] = n_oovo
    Wd[V, O, O, O] = n_oovo.permute(2, 3, 0, 1)
    Wd[V, V, V, O] = n_vvvo
    Wd[V, O, V, V] = n_vvvo.permute(2, 3, 0, 1)
    Fd = F.clone()
    Fd[O, O], Fd[V, V], Fd[V, O] = foo, fvv, r1
    return e0, Fd, Wd


_OPS = {}


def _string_ops(k):
    """Strings of k electrons in 2k orbitals (ascending bit mask), E_pq among them, and the operator
    table over spin-symmetric determinant pairs: rows h'_pq (4 k^2), then W_pqrs (16 k^4)."""
    if k in _OPS:
        return _OPS[k]
    no = 2 * k
    masks = sorted(sum(1 << p for p in c) for c in itertools.combinations(range(no), k))
    at = {m: i for i, m in enumerate(masks)}
    ns = len(masks)
    E = torch.zeros((no, no, ns, ns), dtype=torch.float64)
    for m in masks:
        for q in range(no):
            if not m >> q & 1:
                continue
            m1, s1 = m & ~(1 << q), bin(m & ((1 << q) - 1)).count("1")
            for p in range(no):
                if m1 >> p & 1:
                    continue
                s2 = bin(m1 & ((1 << p) - 1)).count("1")
                E[p, q, at[m1 | 1 << p], at[m]] = (-1.0) ** (s1 + s2)
    E = E.cuda()
    # spin-symmetric basis: (I I), and (I J + J I) / sqrt 2 for I < J
    pairs = [(i, j) for i in range(ns) for j in range(i, ns)]
    P = torch.zeros((ns * ns, len(pairs)), dtype=torch.float64, device="cuda")
    for c, (i, j) in enumerate(pairs):
        if i == j:
            P[i * ns + i, c] = 1.0
        else:
            P[i * ns + j, c] = P[j * ns + i, c] = math.sqrt(0.5)
    eye = torch.eye(ns, dtype=torch.float64, device="cuda")
    one = [P.T @ (torch.kron(E[p, q], eye) + torch.kron(eye, E[p, q])) @ P for p in range(no) for q in range(no)]
    two = []
    for p, q, r, s in itertools.product(range(no), repeat=4):
        ee = 0.5 * (E[p, q] @ E[r, s])
        two.append(P.T @ (torch.kron(ee, eye) + torch.kron(eye, ee) + torch.kron(E[p, q], E[r, s])) @ P)
    table = torch.stack([m.reshape(-1) for m in one + two])
    # determinants of the singles and doubles amplitudes, with their signs
    ref = masks[0]
    def single(i, a):
        return E[k + a, i, :, 0].nonzero().item(), float(E[k + a, i, :, 0].sum())
    assert ref == (1 << k) - 1
    ia = [[single(i, a) for a in range(k)] for i in range(k)]
    col = {pq: c for c, pq in enumerate(pairs)}
    _OPS[k] = (table, ia, col, len(pairs))
    return _OPS[k]


def _solve64(e0, F, W, sp, k):
    """Energies and increments X1[b, i, a], X2[b, i, j, a, b'] of the spaces' Phi-dominant roots."""
    table, ia, col, m = _string_ops(k)
    out_e, out_1, out_2 = [], [], []
    step = 512 if k == 3 else 8192
    for at in range(0, len(sp), step):
        orb = torch.from_numpy(sp[at:at + step, 2:2 + 2 * k].astype(np.int64)).cuda()
        b = len(orb)
        o = [orb.reshape((b,) + tuple(2 * k if d == a else 1 for d in range(4))) for a in range(4)]
        w = W[o[0], o[1], o[2], o[3]]
        f = F[orb[:, :, None], orb[:, None, :]]
        occ = slice(0, k)
        hv = f - 2 * torch.einsum("bpqkk->bpq", w[:, :, :, occ, occ]) + torch.einsum("bpkkq->bpq", w[:, :, occ, occ, :])
        core = e0 - torch.einsum("bkk->b", hv[:, occ, occ]) - torch.einsum("bkk->b", f[:, occ, occ])
        hp = hv - 0.5 * torch.einsum("bprrq->bpq", w)
        H = (torch.cat([hp.reshape(b, -1), w.reshape(b, -1)], 1) @ table).reshape(b, m, m)
        z, e = torch.zeros((b, m - 1), dtype=torch.float64, device="cuda"), H[:, 0, 0].clone()
        if m > 1:
            a, row, colv = H[:, 1:, 1:], H[:, 0, 1:], H[:, 1:, 0]
            eye = torch.eye(m - 1, dtype=torch.float64, device="cuda")
            sh = e
            for outer in range(2):  # (A - e) z = -c with e = H_00 + r z, the factors kept over the inner steps
                lu, piv = torch.linalg.lu_factor(a - sh[:, None, None] * eye)
                for _ in range(8):
                    res = colv + torch.einsum("bij,bj->bi", a, z) - e[:, None] * z
                    z = z - torch.linalg.lu_solve(lu, piv, res[:, :, None])[:, :, 0]
                    e = H[:, 0, 0] + (row * z).sum(1)
                sh = e
            res = (colv + torch.einsum("bij,bj->bi", a, z) - e[:, None] * z).norm(dim=1)
            for i in torch.nonzero(~((res < 1e-11) & (z.norm(dim=1) < 0.9))).flatten().tolist():
                ev, vec = np.linalg.eig(H[i].cpu().numpy())
                j = int(np.argmax(np.abs(vec[0])))
                e[i] = float(ev[j].real)
                z[i] = torch.from_numpy((vec[1:, j] / vec[0, j]).real.copy()).cuda()
        c = torch.cat([torch.ones((b, 1), dtype=torch.float64, device="cuda"), z], 1)
        x1 = torch.zeros((b, k, k), dtype=torch.float64, device="cuda")
        cab = torch.zeros((b, k, k, k, k), dtype=torch.float64, device="cuda")
        rt = math.sqrt(0.5)
        for i, a_ in itertools.product(range(k), repeat=2):
            s, sg = ia[i][a_]
            x1[:, i, a_] = sg * rt * c[:, col[(0, s)]]
            for j, b_ in itertools.product(range(k), repeat=2):
                t, tg = ia[j][b_]
                cab[:, i, j, a_, b_] = sg * tg * c[:, col[(min(s, t), max(s, t))]] * (1.0 if s == t else rt)
        x2 = cab - torch.einsum("bia,bjc->bijac", x1, x1)
        out_e.append((core + e).cpu().numpy())
        out_1.append(x1.cpu().numpy())
        out_2.append((0.5 * (x2 + x2.permute(0, 2, 1, 4, 3))).cpu().numpy())
    return np.concatenate(out_e), np.concatenate(out_1), np.concatenate(out_2)


def _order(eps, sp):
    """Positions of the spaces by ascending Delta-eps (ties: size, then orbital tuple)."""
    d = np.zeros(len(sp))
    for i, r in enumerate(sp):
        k = r[0]
        d[i] = sum(eps[q] for q in r[2 + k:2 + 2 * k]) - sum(eps[q] for q in r[2:2 + k])
    return np.lexsort(tuple(sp[:, c] for c in range(7, 1, -1)) + (sp[:, 0], d))


def _sweep64(e0, F, W, sp, o, v, t1, t2):
    """Energies of the ordered spaces and the pool in which every amplitude took its first space's increment."""
    energy = np.zeros(len(sp))
    first1, first2 = np.full(t1.size, len(sp)), np.full(t2.size, len(sp))
    parts = []
    for k in (1, 2, 3):
        at = np.nonzero(sp[:, 0] == k)[0]
        if not len(at):
            continue
        energy[at], x1, x2 = _solve64(e0, F, W, sp[at], k)
        occ, vir = sp[at, 2:2 + k].astype(np.int64), sp[at, 2 + k:2 + 2 * k].astype(np.int64) - o
        i1 = occ[:, :, None] * v + vir[:, None, :]
        i2 = ((occ[:, :, None, None, None] * o + occ[:, None, :, None, None]) * v + vir[:, None, None, :, None]) * v + vir[:, None, None, None, :]
        s1, s2 = np.broadcast_to(at[:, None, None], i1.shape), np.broadcast_to(at[:, None, None, None, None], i2.shape)
        np.minimum.at(first1, i1, s1)
        np.minimum.at(first2, i2, s2)
        parts.append((i1, s1, x1, i2, s2, x2))
    n1, n2 = t1.copy().reshape(-1), t2.copy().reshape(-1)
    for i1, s1, x1, i2, s2, x2 in parts:
        m1, m2 = first1[i1] == s1, first2[i2] == s2
        n1[i1[m1]] += x1[m1]
        n2[i2[m2]] += x2[m2]
    return energy, n1.reshape(t1.shape), n2.reshape(t2.shape)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("train", "infer"):
        p, x, t = (torch.from_numpy(a.astype(np.float64)).cuda() for a in _net(case, seed))
        nin, nout, H = qflow.MLP_NIN, qflow.MLP_NOUT, case["hidden"]
        p.requires_grad_(kind == "train")
        w1, b1, w2, b2, w3, b3 = torch.split(p, [nin * H, H, H * H, H, H * nout, nout])
        y = torch.tanh(torch.tanh(x @ w1.reshape(nin, H) + b1) @ w2.reshape(H, H) + b2) @ w3.reshape(H, nout) + b3
        if kind == "infer":
            return {"y": y}
        loss = ((y - t) ** 2).sum() / (2 * case["rows"])
        g, = torch.autograd.grad(loss, p)
        p = p.detach()
        new = p - float(np.float32(2e-3)) * g / (g.abs() + float(np.float32(1e-8)))
        one = lambda b: 1.0 - float(np.float32(b))  # noqa: E731
        return {"loss": loss.detach().reshape(1), "grad": g, "m": one(0.9) * g, "v": one(0.999) * g * g, "params": new}
    n, o = case["n"], case["nocc"]
    v = n - o
    eps, h, eri = _system(case, seed)
    if kind == "dress":
        t1, t2 = synth.random_amplitudes(o, v, seed, 0.01, 0.02)
        e0, F, W = _dress64(_cuda(h), _cuda(eri), _cuda(t1), _cuda(t2), o)
        return {"e0": e0.reshape(1), "F": F, "W": W}
    if kind == "solve":
        t1, t2 = synth.random_amplitudes(o, v, seed, 0.01, 0.02)
        sp = _class_spaces(case, seed + 1)
        sp = sp[_order(eps, sp)]
        e0, F, W = _dress64(_cuda(h), _cuda(eri), _cuda(np.zeros_like(t1)), _cuda(np.zeros_like(t2)), o)
        energy, n1, n2 = _sweep64(e0, F, W, sp, o, v, t1, t2)
        return {"energy": energy, "status": None, "t1": n1, "t2": n2}
    if case["form"] != "ses" or n > 48:  # the Hermitian form and the large systems take too long this way
        return None
    sp = _space_list(case, eps, seed + 1)
    if len(sp) > 70000 or np.count_nonzero(sp[:, 0] == 3) > 20000:
        return None
    sp = sp[_order(eps, sp)]
    t1, t2 = np.zeros((o, v)), np.zeros((o, o, v, v))
    hd, gd = _cuda(h), _cuda(eri)
    for _ in range(3):  # two sweeps make the pool, the third is the measured one
        energy, t1, t2 = _sweep64(*_dress64(hd, gd, _cuda(t1), _cuda(t2), o), sp, o, v, t1, t2)
    return {"mean": float(energy.mean()), "energies": energy, "nfailed": None, "t1": t1, "t2": t2}
