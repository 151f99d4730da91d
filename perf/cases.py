"""The work that performance is measured on: index -> plan -> merge through the package's public calls.

A case is one checkpoint family (tensor shapes, data type, number of experts, block size), one
operator and one way to use the three calls:

* "step"      the experts are new: catalog (mp_index_blocks), then a plan and a merge per budget;
* "merge"     the catalog is kept from earlier (it is reusable), each pass plans and merges;
* "import"    the catalog comes from saved statistics, some entries missing (tensor-level
              fallback): mp_index_import, plan, merge;
* "validated" a touched-only merge with the catalog's block hashes: the inputs that were read
              are validated and the output's hashes recorded;
* "catalog"   the catalog alone, exported with mp_index_stats.

Every pass reads its manifests (realized reads, touched blocks, plan digest) and frees its
handles, as a program does that merges and goes on.  The families are random: a base of
0.02 * normal values and experts that differ from it by a scale per (expert, block), lognormal
on an active share of the blocks and 1e-7 elsewhere (which bf16 storage rounds to exact zeros
but for a few elements near zero).
"""
import math

import numpy as np
import torch

import paper_2605_29489_gb300 as mp

KINDS = {"avg": mp.MP_OP_AVG, "ta": mp.MP_OP_TA, "ties": mp.MP_OP_TIES, "dare": mp.MP_OP_DARE,
         "avg_renorm": mp.MP_OP_AVG_RENORM, "dare_ties": mp.MP_OP_DARE_TIES, "ties_masked": mp.MP_OP_TIES_MASKED}


def _case(name, shape, op, mode, budgets, K, dtype="bf16", block=65536, layers=0, active=0.3, per_expert=False,
          log_mu=math.log(1e-3), log_sigma=1.0, density=0.2, trim_scope=0, drop_p=0.9, lam=1.0, host_pool=False,
          score_mode=0, params=0, tensors=0):
    c = dict(shape=shape, layers=layers, params=params, tensors=tensors, dtype=dtype, block=block, K=K, op=op, mode=mode,
             budgets=",".join(str(f) for f in budgets), active=active, per_expert=per_expert, log_mu=log_mu,
             log_sigma=log_sigma, density=density, trim_scope=trim_scope, drop_p=drop_p, lam=lam, host_pool=host_pool,
             score_mode=score_mode)
    return dict(c, name=name) if name else c


def listed():
    llama = dict(log_mu=math.log(2e-4), log_sigma=1.2, active=0.4)
    return [
        # a toy or adapter-sized family, swept over budgets: launches and latency count
        _case("tiny-fp32-avg-sweep", "square512", "avg", "step", (1.0, 0.5, 0.25), 4, "fp32", 4096, layers=8),
        # a handful of ragged tensors (biases, norms, odd matrices), one TIES merge
        _case("ragged-bf16-ties", "mix", "ties", "step", (0.5,), 3, block=4096, params=1500001, tensors=11, active=0.5),
        # a small language model: task arithmetic swept over the usual budgets
        _case("qwen05b-ta-sweep", "qwen2.5-0.5b", "ta", "step", (1.0, 0.5, 0.25, 0.1), 8, layers=24, lam=0.3),
        # the same from a saved catalog with missing entries, averaged over the selected experts
        _case("qwen05b-renorm-import", "qwen2.5-0.5b", "avg_renorm", "import", (0.5,), 8, layers=24),
        # many experts (over eight), a budget, catalog at hand
        _case("qwen05b-ties-k16-merge", "qwen2.5-0.5b", "ties", "merge", (0.25,), 16, layers=24),
        # touched-only output with input validation and output hashes
        _case("qwen05b-touched-validated", "qwen2.5-0.5b", "ta", "validated", (0.25,), 4, layers=24, lam=0.3),
        # experts in host memory, only the planned blocks brought in
        _case("qwen05b-2l-hostpool-avg", "qwen2.5-0.5b", "avg", "step", (0.25,), 4, layers=2, host_pool=True),
        # sixteen experts of a mid-size model, random drop and rescale, from new experts to the merge
        _case("qwen15b-dare-step", "qwen2.5-1.5b", "dare", "step", (0.25,), 16, layers=28, active=0.25, per_expert=True),
        # the same experts with sign election, catalog at hand
        _case("qwen15b-dare-ties-merge", "qwen2.5-1.5b", "dare_ties", "merge", (0.25,), 16, layers=28, active=0.25,
              per_expert=True),
        # fp32 checkpoints (one large transformer layer), one trim population per expert
        _case("llama1l-fp32-ties", "llama-3-8b", "ties", "step", (1.0,), 4, "fp32", layers=1, trim_scope=1, **llama),
        # TIES applied after masking: the threshold is found anew for each plan
        _case("llama2l-ties-masked", "llama-3-8b", "ties_masked", "step", (0.5,), 4, layers=2, **llama),
        # the large one: eight layers of an 8B model (more would not fit three times), TIES over the budgets
        _case("llama8l-ties-sweep", "llama-3-8b", "ties", "step", (1.0, 0.5, 0.25, 0.1), 4, layers=8, **llama),
    ]


def draw(rng):
    """One more family: sizes over the whole range, ragged tensors, every operator, type and mode."""
    op = rng.choice(sorted(KINDS))
    dtype = rng.choice(("bf16", "bf16", "bf16", "fp32"))
    es = 2 if dtype == "bf16" else 4
    K = rng.choice((1, 2, 3, 4, 4, 5, 7, 8, 8, 11, 16, 20, 32))
    host_pool = op != "ties_masked" and rng.random() < 0.1
    # elements of one checkpoint: 2^17 up to what keeps the state below 16 GB (1 GB in host memory)
    top = (1e9 if host_pool else 16e9) / ((K + 2) * es)
    n = int(math.exp(rng.uniform(math.log(1 << 17), math.log(top))))
    big = n > 20_000_000
    modes = ["step", "merge", "catalog"]
    if not host_pool:
        modes.append("validated")
    if op != "ties_masked":
        modes.append("import")
    mode = rng.choice(modes)
    block = rng.choice((65536, 65536, 40000)) if big else rng.choice((4096, 4096, 16384, 1000))
    nb = rng.choice((1, 1, 2)) if mode in ("step", "merge") else 1
    budgets = sorted((round(rng.choice((1.0, rng.uniform(0.05, 1.0))), 3) for _ in range(nb)), reverse=True)
    return _case(None, "mix", op, mode, budgets, K, dtype, block, params=n, tensors=rng.randint(5, 300),
                 active=rng.choice((0.25, 0.3, 0.4, 0.6)), per_expert=rng.random() < 0.4,
                 density=rng.choice((0.1, 0.2, 0.35, 0.5)), trim_scope=rng.choice((0, 0, 1)),
                 drop_p=rng.choice((0.5, 0.9, 0.95)), lam=rng.choice((0.3, 0.7, 1.0)), host_pool=host_pool,
                 score_mode=rng.choice((0, 0, 1)))


# ---- shapes ---------------------------------------------------------------------------------------

def _decoder(hidden, layers, kv, inter, vocab, bias, head):
    t = [vocab * hidden] if vocab else []
    for _ in range(layers):
        t.append(hidden)
        for out in (hidden, kv, kv):
            t.append(out * hidden)
            if bias:
                t.append(out)
        t += [hidden * hidden, hidden, inter * hidden, inter * hidden, hidden * inter]
    return t + [hidden] + ([vocab * hidden] if head else [])


def _numels(c):
    s, layers = c["shape"], c["layers"]
    if s == "square512":
        return [512 * 512] * layers
    if s == "qwen2.5-0.5b":
        return _decoder(896, layers, 128, 4864, 151936, True, False)
    if s == "qwen2.5-1.5b":
        return _decoder(1536, layers, 256, 8960, 151936, True, False)
    if s == "llama-3-8b":  # transformer layers only
        return _decoder(4096, layers, 1024, 14336, 0, False, False)
    # "mix": ragged tensors, a few of them large and many small, `params` elements in all
    w = [math.exp(-0.05 * k) * (0.02 if k % 3 == 2 else 1.0) for k in range(c["tensors"])]
    per = c["params"] / sum(w)
    return [max(3, int(per * x) | (k & 1)) for k, x in enumerate(w)]


def _layout(c):
    """(offsets, numels, total): each tensor starts on a 16-byte boundary"""
    al = 8 if c["dtype"] == "bf16" else 4
    offs, nums, off = [], _numels(c), 0
    for n in nums:
        offs.append(off)
        off = (off + n + al - 1) // al * al
    return offs, nums, off


def _blocks(c):
    """(start, length, tensor) of every block, in tensor order"""
    offs, nums, _ = _layout(c)
    E = c["block"]
    st, ln, tn = [], [], []
    for t, (o, n) in enumerate(zip(offs, nums)):
        s = np.arange(0, n, E, dtype=np.int64)
        st.append(o + s)
        ln.append(np.minimum(E, n - s))
        tn.append(np.full(s.size, t, np.int64))
    return np.concatenate(st), np.concatenate(ln), np.concatenate(tn)


def _windows(starts, total, most=1 << 26):
    """runs of consecutive blocks [b0, b1) of about `most` elements, and their element range"""
    ends = np.append(starts[1:], total)
    b0 = 0
    while b0 < starts.size:
        b1 = max(b0 + 1, int(np.searchsorted(ends, starts[b0] + most, side="right")))
        yield b0, b1, int(starts[b0]), int(ends[b1 - 1])
        b0 = b1


# ---- inputs ---------------------------------------------------------------------------------------

def _inputs(c, seed, device="cuda"):
    """(base, [experts]) as flat tensors on the GPU"""
    starts, lens, _ = _blocks(c)
    total = _layout(c)[2]
    nb, K = starts.size, c["K"]
    dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    r = np.random.default_rng([int(seed), 17])
    n_act = int(c["active"] * nb)
    scales = np.full((K, nb), 1e-7, np.float32)
    shared = r.permutation(nb)[:n_act]
    for i in range(K):
        on = r.permutation(nb)[:n_act] if c["per_expert"] else shared
        scales[i, on] = np.exp(r.normal(c["log_mu"], c["log_sigma"], n_act))
    ext = torch.from_numpy(np.diff(np.append(starts, total))).to(device)
    sc = torch.from_numpy(scales).to(device)
    g = torch.Generator(device=device)
    g.manual_seed(int(seed) * 1000003 + 12345)
    base = torch.empty(total, dtype=dt, device=device)
    experts = [torch.empty(total, dtype=dt, device=device) for _ in range(K)]
    for b0, b1, e0, e1 in _windows(starts, total):
        n = e1 - e0
        base[e0:e1] = torch.randn(n, generator=g, device=device) * 0.02
        w = base[e0:e1].float()
        for i in range(K):
            s = torch.repeat_interleave(sc[i, b0:b1], ext[b0:b1], output_size=n)
            experts[i][e0:e1] = torch.addcmul(w, s, torch.randn(n, generator=g, device=device))
    return base, experts


def _coefs(c):
    K = c["K"]
    return [c["lam"]] * K if c["op"] == "ta" else [1.0 / K] * K


def _missing(c, seed):
    """which entries a saved catalog lacks: a tenth of the (expert, tensor) pairs and a few others"""
    _, _, tn = _blocks(c)
    r = np.random.default_rng([int(seed), 29])
    pairs = r.random((c["K"], int(tn[-1]) + 1)) < 0.1
    return pairs[:, tn] | (r.random((c["K"], tn.size)) < 0.001)


def _budgets(c):
    return [float(f) for f in c["budgets"].split(",")]


def prepare(case, seed):
    c = dict(case)
    base, experts = _inputs(c, seed)
    offs, nums, _ = _layout(c)
    if c["host_pool"]:
        experts = [e.cpu().pin_memory() for e in experts]
    fam = mp.family(list(zip(offs, nums)), base, experts, block_elems=c["block"],
                    dtype=mp.MP_BF16 if c["dtype"] == "bf16" else mp.MP_F32, experts_location=1 if c["host_pool"] else 0)
    op = mp.make_op(KINDS[c["op"]], alpha=_coefs(c), lam=c["lam"], density=c["density"], trim_scope=c["trim_scope"],
                    drop_p=c["drop_p"], seed=2605 + int(seed), score_mode=c["score_mode"])
    s = dict(c=c, fam=fam, op=op, B=[mp.mp_budget_from_fraction(fam, f) for f in _budgets(c)])
    if c["mode"] != "catalog":
        s["outs"] = [base.clone() if c["mode"] == "validated" else torch.zeros_like(base) for _ in s["B"]]
    if c["mode"] == "merge":
        s["idx"] = mp.mp_index_blocks(fam, op)
    if c["mode"] == "import":
        with mp.mp_index_blocks(fam, op) as idx:
            norm, maxabs, nnz, tau = mp.mp_index_stats(idx)
        nnz[_missing(c, seed)] = mp.MP_NNZ_MISSING
        s["saved"] = (norm, maxabs, nnz, tau if c["op"] == "ties" else None)
    return s


def _manifest(s, man):
    m = mp.mp_manifest_info(man, s["c"]["K"])
    return {"realized": m["realized"].view(np.int64), "touched": m["touched"],
            "digest": [m["digest"] >> 32, m["digest"] & 0xFFFFFFFF]}


def run(state):
    s = state
    fam, op, mode = s["fam"], s["op"], s["c"]["mode"]
    if mode == "merge":
        idx = s["idx"]
    elif mode == "import":
        idx = mp.mp_index_import(fam, op, *s["saved"])
    else:
        idx = mp.mp_index_blocks(fam, op)
    if mode == "catalog":
        norm, maxabs, nnz, tau = mp.mp_index_stats(idx)
        idx.free()
        return {"norm": norm, "maxabs": maxabs, "nnz": nnz.astype(np.int64), "tau": tau.astype(np.int64)}
    if mode == "validated":
        mp.mp_index_hashes(fam, idx)
    merge = mp.mp_merge_touched if mode == "validated" else mp.mp_merge
    made = []
    for B, out in zip(s["B"], s["outs"]):
        plan = mp.mp_plan(idx, op, B)
        made.append((plan, merge(fam, idx, plan, out)))
    res = {"merged": list(s["outs"])}
    if mode == "validated":
        plan, man = made[0]
        mp.mp_manifest_validate(fam, idx, plan, s["outs"][0], man)
        v = mp.mp_manifest_validation(man, mp.mp_index_shape(idx)[0])
        res["out_hash"] = v["out_hash"].view(np.int64)
        res["validation"] = [v["checked"], v["mismatched"]]
    res["manifest"] = [_manifest(s, man) for _, man in made]
    for plan, man in made:
        man.free()
        plan.free()
    if mode != "merge":
        idx.free()
    return res


# ---- what a pass cannot do without ----------------------------------------------------------------

def work(case):
    """The catalog reads the base and every expert once; a merge reads the base (or its touched
    blocks) and the planned expert blocks once and writes as much as it merges; hashing reads
    what it hashes.  TIES plans hold about the active share of the experts at most."""
    c = case
    n, K = sum(_numels(c)), c["K"]
    es = 2 if c["dtype"] == "bf16" else 4
    one, mode = n * es, c["mode"]
    nbytes, flops = 0.0, 0.0
    if mode in ("step", "catalog", "validated"):
        nbytes += (K + 1) * one
        flops += 4.0 * n * K
    if mode != "catalog":
        for f in _budgets(c):
            sel = min(f, c["active"]) if c["op"] == "ties" and mode != "import" else f
            touched = min(1.0, f * K) if mode == "validated" else 1.0
            if mode == "validated" and not c["per_expert"]:
                touched = f
            nbytes += 2 * touched * one + sel * K * one
            flops += 3.0 * sel * K * n
            if mode == "validated":
                nbytes += (K + 1) * one + 2 * one + sel * K * one
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # against 64 bits (exact): bf16 results are within 1.2e-3, fp32 within 3e-8 (to 1e-7 with
    # larger deltas); the norms of a catalog (32-bit sums of up to 65,536 squares) within 1.1e-7.  Whole numbers (plans, counts,
    # hashes, thresholds) do not differ.  An output hash would differ with any rounding, so
    # validated merges are compared exactly.
    if case["mode"] == "validated":
        return "exact"
    if case["mode"] == "catalog":
        return {"rel": 5e-7, "max": 5e-6}
    return {"rel": 5e-3, "max": 0.1} if case["dtype"] == "bf16" else {"rel": 5e-7, "max": 1e-4}


# ---- the same results in 64 bits ------------------------------------------------------------------

def _keys(d):
    """TIES's trim key: the bf16 magnitude of the 32-bit delta"""
    return d.abs().to(torch.bfloat16).view(torch.int16).to(torch.int64) & 0x7FFF


def _philox_keep(j0, n, i, seed, p, device):
    """DARE's keep mask of elements j0 .. j0 + n - 1 (j0 a multiple of 8): Philox4x32-10 (Salmon et
    al., 2011), counter (j / 8, expert, "DARE"), 16-bit word j mod 8 >= floor(65536 p)"""
    M = 0xFFFFFFFF
    q = torch.arange(j0 // 8, (j0 + n + 7) // 8, device=device)
    x = [q & M, q >> 32, torch.full_like(q, i), torch.full_like(q, 0x44415245)]
    k0, k1 = seed & M, (seed >> 32) & M

    def mul(m, a):  # high and low halves of the 64-bit product, in 16-bit parts (no overflow)
        lo, hi = (a & 0xFFFF) * m, (a >> 16) * m
        s = (lo >> 16) + hi
        return s >> 16, ((s & 0xFFFF) << 16) | (lo & 0xFFFF)

    for r in range(10):
        h0, l0 = mul(0xD2511F53, x[0])
        h1, l1 = mul(0xCD9E8D57, x[2])
        x = [h1 ^ x[1] ^ ((k0 + r * 0x9E3779B9) & M), l1, h0 ^ x[3] ^ ((k1 + r * 0xBB67AE85) & M), l0]
    w = torch.stack([h for v in x for h in (v & 0xFFFF, v >> 16)], 1).reshape(-1)[:n]
    return w >= math.floor(p * 65536)


def exact(case, seed):
    c = dict(case)
    K, op = c["K"], c["op"]
    starts, lens, tn = _blocks(c)
    total, nb = _layout(c)[2], starts.size
    es = 2 if c["dtype"] == "bf16" else 4
    if c["mode"] == "validated" or total * K > 3e10:
        return None  # the hashes have no 64-bit value; the largest would take too long
    base, experts = _inputs(c, seed)
    d_len = torch.from_numpy(lens).cuda()
    d_ext = torch.from_numpy(np.diff(np.append(starts, total))).cuda()
    wins = list(_windows(starts, total, 1 << 25))

    def window(b0, b1, e0, e1):
        """block of each element of a window (within it), and whether a tensor covers it"""
        blk = torch.repeat_interleave(torch.arange(b1 - b0, device="cuda"), d_ext[b0:b1], output_size=e1 - e0)
        first = torch.cumsum(d_ext[b0:b1], 0) - d_ext[b0:b1]
        live = torch.arange(e1 - e0, device="cuda") - first[blk] < d_len[b0:b1][blk]
        return blk, live

    ties = op in ("ties", "ties_masked")
    grp_of = np.zeros(nb, np.int64) if c["trim_scope"] else tn
    G = int(grp_of[-1]) + 1
    gnum = np.bincount(grp_of, weights=lens, minlength=G).astype(np.int64)
    # the statistics
    ss = torch.zeros(K, nb, dtype=torch.float64, device="cuda")
    mx = torch.zeros(K, nb, dtype=torch.float32, device="cuda")
    nz = torch.zeros(K, nb, dtype=torch.int64, device="cuda")
    for b0, b1, e0, e1 in wins:
        blk, live = window(b0, b1, e0, e1)
        for i in range(K):
            d = torch.where(live, experts[i][e0:e1].float() - base[e0:e1].float(), 0.0)
            n_el = d_ext[b0:b1]
            ss[i, b0:b1] = torch.segment_reduce(d.double() ** 2, "sum", lengths=n_el)
            mx[i, b0:b1] = torch.segment_reduce(d.abs(), "max", lengths=n_el)
            nz[i, b0:b1] = torch.segment_reduce((d != 0).double(), "sum", lengths=n_el).long()
    norm = ss.sqrt().cpu().numpy()

    def thresholds(mask):
        """the k-th largest key of each (expert, group); an omitted block counts as zeros"""
        tau = np.zeros((K, G), np.int64)
        for i in range(K):
            h = np.zeros((G, 32768), np.int64)
            for b0, b1, e0, e1 in wins:
                blk, live = window(b0, b1, e0, e1)
                key = _keys(experts[i][e0:e1].float() - base[e0:e1].float())
                if mask is not None:
                    key = key * torch.from_numpy(mask[i, b0:b1]).cuda()[blk]
                g = grp_of[b0:b1] - grp_of[b0]
                gg = torch.from_numpy(g).cuda()[blk]
                n_g = int(g[-1]) + 1
                h[grp_of[b0]:grp_of[b0] + n_g] += torch.bincount((gg * 32768 + key)[live], minlength=n_g * 32768).view(
                    n_g, 32768).cpu().numpy()
            for q in range(G):
                k = math.floor(float(np.float32(c["density"])) * int(gnum[q]))
                cum = np.cumsum(h[q][::-1])
                tau[i, q] = 0x8000 if k == 0 else 32767 - int(np.searchsorted(cum, k))
        return tau

    tau = thresholds(None) if op == "ties" or (ties and c["mode"] == "catalog") else None
    if c["mode"] == "catalog":
        return {"norm": norm, "maxabs": mx.double().cpu().numpy(), "nnz": None, "tau": None}
    mxk = _keys(mx).cpu().numpy()
    nnz = nz.cpu().numpy()
    cand = nnz > 0
    if op == "ties":
        cand &= mxk >= tau[:, grp_of]
    coef = [abs(c["lam"])] * K if op in ("ties", "dare_ties", "ties_masked") else [abs(a) for a in _coefs(c)]
    score = np.array(coef, np.float64)[:, None] * norm
    cost = np.broadcast_to(lens * es, (K, nb))
    # units: (score, cost, unit id, expert, its blocks)
    iu, bu = np.nonzero(cand)
    units = None
    if c["mode"] == "import":
        gone = _missing(c, seed)
        first = np.searchsorted(tn, np.arange(int(tn[-1]) + 2))
        whole = np.zeros((K, int(tn[-1]) + 1), bool)
        np.logical_or.at(whole, (np.nonzero(gone)[0], tn[np.nonzero(gone)[1]]), True)
        keep = ~whole[iu, tn[bu]]
        iu, bu = iu[keep], bu[keep]
        known = np.where(gone, 0.0, norm)
        wi, wt = np.nonzero(whole)
        w_norm = np.array([math.sqrt((known[i, first[t]:first[t + 1]] ** 2).sum()) for i, t in zip(wi, wt)])
        w_cost = np.array([int(lens[first[t]:first[t + 1]].sum()) * es for t in wt], np.int64)
        units = (wi, wt, w_norm * np.array(coef)[wi], w_cost, first)
    sc, co, ui = score[iu, bu], cost[iu, bu], bu * K + iu
    who = np.arange(iu.size)
    if units is not None:
        wi, wt, w_sc, w_cost, first = units
        sc, co = np.concatenate([sc, w_sc]), np.concatenate([co, w_cost])
        ui = np.concatenate([ui, first[wt] * K + wi])
        who = np.arange(sc.size)
    if c["score_mode"]:
        sc = sc / co
    order = who[np.lexsort((ui, -sc.astype(np.float32)))]
    offs, nums, _ = _layout(c)
    merged = []
    for f in _budgets(c):
        B, taken = math.floor(f * (K * sum(nums) * es)), 0
        mask = np.zeros((K, nb), bool)
        smallest = int(co.min()) if co.size else 0
        for u in order.tolist():
            if taken + int(co[u]) > B:
                if B - taken < smallest:
                    break
                continue
            taken += int(co[u])
            if u < iu.size:
                mask[iu[u], bu[u]] = True
            else:
                i, t = int(wi[u - iu.size]), int(wt[u - iu.size])
                mask[i, first[t]:first[t + 1]] = True
        th = thresholds(mask) if op == "ties_masked" else tau
        d_mask = torch.from_numpy(mask).cuda()
        out = torch.zeros(total, dtype=torch.float64, device="cuda")
        for b0, b1, e0, e1 in wins:
            blk, live = window(b0, b1, e0, e1)
            x0 = base[e0:e1].double()
            acc = torch.zeros_like(x0)
            P, N = torch.zeros_like(x0), torch.zeros_like(x0)
            cp, cn = torch.zeros_like(blk), torch.zeros_like(blk)
            if op == "avg_renorm":  # counted: selected, or known from the catalog to be zero
                zero = nnz[:, b0:b1] == 0
                if c["mode"] == "import":
                    zero &= ~gone[:, b0:b1]
                cnt = mask[:, b0:b1] | zero
                den = torch.from_numpy((cnt * np.array(_coefs(c))[:, None]).sum(0)).cuda()[blk].clamp_min(1e-300)
            for i in range(K):
                if not mask[i, b0:b1].any():
                    continue
                sel = d_mask[i, b0:b1][blk]
                d = experts[i][e0:e1].double() - x0
                if op in ("dare", "dare_ties"):
                    keep = _philox_keep(e0, e1 - e0, i, 2605 + int(seed), c["drop_p"], "cuda")
                    d = torch.where(keep & sel, d / (1.0 - c["drop_p"]), 0.0)
                elif ties:
                    t_e = torch.from_numpy(th[i, grp_of[b0:b1]]).cuda()[blk]
                    key = _keys(experts[i][e0:e1].float() - base[e0:e1].float())
                    d = torch.where(sel & (key >= t_e), d, 0.0)
                else:
                    d = torch.where(sel, d, 0.0)
                if ties or op == "dare_ties":
                    P += d.clamp_min(0)
                    N += d.clamp_max(0)
                    cp += d > 0
                    cn += d < 0
                elif op == "avg_renorm":
                    acc += d * _coefs(c)[i] / den
                else:
                    acc += d * _coefs(c)[i]
            if ties or op == "dare_ties":
                acc = torch.where(P > -N, P / cp.clamp_min(1), torch.where(P < -N, N / cn.clamp_min(1), 0.0)) * c["lam"]
            out[e0:e1] = torch.where(live, x0 + acc, 0.0)
        merged.append(out)
    none = {"realized": None, "touched": None, "digest": [None, None]}
    return {"merged": merged, "manifest": [none for _ in merged]}
