"""Performance cases: what users of the library have it do, through its public entry points.

Every case is one call (or one burst of calls) of the Python binding on device
buffers, or on pinned host buffers for the host-stream case.  Rings, levels and
batch sizes are those of the presets, the benchmark and the tests.  Ciphertext
and key residues are uniform modulo their primes, which is how encryptions and
evaluation keys look to the arithmetic.

All outputs are residues or integer words (whole numbers, equal word for word
in every build), so `exact` has no floating-point reference to give.
"""
import weakref

import numpy as np
import torch

import paper_2003_04510_gb300 as he

DEV = "cuda"

# Rings: (logN, L, K, alpha, q_bits, p_bits, h).  n12..n17 are the library's presets.  n13 and n14 fill
# the gap between them; n16_d8 cuts the chain into eight digits of three limbs (a smaller key switch basis).
RINGS = {
    "n12": (12, 3, 1, 1, 50, 51, 64),
    "n13": (13, 6, 2, 2, 50, 51, 64),
    "n14": (14, 9, 4, 4, 50, 51, 64),
    "n15": (15, 16, 8, 8, 54, 55, 192),
    "n16": (16, 24, 8, 8, 54, 55, 192),
    "n16_d8": (16, 24, 3, 3, 54, 55, 192),
    "n17": (17, 44, 12, 11, 54, 54, 192),
}

# Launch shapes (he_shape's fields in order).  "default" is a context as created.  The others are what
# he_autotune settles on for the benchmark's workloads, set once per context as a tuned program does.
SHAPES = {
    "default": None,
    "tuned_single": (1, 8, 2, 15, 8, 7, 1, 1, 0),
    "tuned_large": (2, 8, 1, 15, 8, 7, 1, 0, 0),
    "tuned_batch": (2, 16, 2, 15, 8, 3, 1, 0, 0),
}


def batch_levels(count, lo, hi, seed):
    return [int(v) for v in np.random.Generator(np.random.PCG64(seed)).integers(lo, hi + 1, size=count)]


def listed():
    return [
        # The smallest call: a toy ring, three limbs, one digit per limb.  Latency and launches.
        {"name": "mul_n12", "kind": "single", "ring": "n12", "call": "mul_rescale", "level": 3, "shape": "default"},
        # The serving mix's common ring at an odd level whose last digit holds one limb.
        {"name": "mul_n15", "kind": "single", "ring": "n15", "call": "mul_rescale", "level": 9, "shape": "default"},
        # The headline workload: one HE Mul + rescale at N = 2^16 from the top of the chain, tuned once.
        {"name": "mul_n16", "kind": "single", "ring": "n16", "call": "mul_rescale", "level": 24,
         "shape": "tuned_single"},
        # The same at N = 2^17, 44 limbs, four digits: the largest single call.
        {"name": "mul_n17", "kind": "single", "ring": "n17", "call": "mul_rescale", "level": 44,
         "shape": "tuned_large"},
        # A rotation (the plain mod down without rescale) in the middle of the chain.
        {"name": "rotate_n16", "kind": "single", "ring": "n16", "call": "rotate", "level": 13, "shape": "default"},
        # A plaintext-weighted sum between multiplications: two plaintext products, a sum, a rescale.
        {"name": "weighted_sum_n16", "kind": "linear", "ring": "n16", "level": 17},
        # 64 independent HE Muls at uneven levels as one batch (the batched benchmark's jobs).
        {"name": "batch_n16", "kind": "batch", "ring": "n16", "levels_lo": 4, "levels_hi": 24, "jobs": 64,
         "levels_seed": 1604, "shape": "tuned_batch"},
        # A small batch replayed from a captured graph.
        {"name": "graph_n15", "kind": "graph", "ring": "n15", "levels_lo": 2, "levels_hi": 16, "jobs": 16,
         "levels_seed": 1502},
        # A burst of requests of both serving rings through the continuous-batching server.
        {"name": "serve_mix", "kind": "serve", "jobs": 48, "levels_seed": 1503},
        # A run of jobs whose operands and results live in pinned host memory.
        {"name": "host_stream_n16", "kind": "host", "ring": "n16", "jobs": 4, "levels_lo": 9, "levels_hi": 24,
         "levels_seed": 1605},
        # The paper's own HE Mul on BigInt coefficients at its parameters.
        {"name": "bigint_mul_n16", "kind": "bigint", "logN": 16, "logQ": 1200, "logp": 30, "logq": 1200},
        # The same at a small ring and a modulus that is no multiple of the word, followed by its rescale.
        {"name": "bigint_mul_n12", "kind": "bigint", "logN": 12, "logQ": 300, "logp": 30, "logq": 250},
    ]


def draw(rng):
    """One more case of the ranges above; none costs more than the 64-job batch."""
    kind = rng.choice(["single", "single", "single", "linear", "batch", "graph", "bigint"])
    ring = rng.choice(sorted(RINGS))
    L = RINGS[ring][1]
    if kind == "single":
        call = rng.choice(["mul_rescale", "mul_rescale", "mul_rescale_pq", "mul", "rotate", "mul_rescale_seeded"])
        lo = 1 if call in ("mul", "rotate") else 2
        shapes = ["default"] + (["tuned_single", "tuned_large"] if ring in ("n16", "n17") else [])
        return {"kind": kind, "ring": ring, "call": call, "level": rng.randint(lo, L), "shape": rng.choice(shapes)}
    if kind == "linear":
        return {"kind": kind, "ring": ring, "level": rng.randint(2, L)}
    if kind == "bigint":
        logN, logQ = rng.randint(12, 16), rng.randint(128, 1216)
        return {"kind": kind, "logN": logN, "logQ": logQ, "logp": 30, "logq": rng.randint(64, logQ)}
    ring = rng.choice([r for r in sorted(RINGS) if r != "n17"])
    L = RINGS[ring][1]
    lo = rng.randint(2, max(2, L - 1))
    case = {"kind": kind, "ring": ring, "levels_lo": lo, "levels_hi": rng.randint(lo, L),
            "jobs": int(2 ** rng.uniform(0, 5)) if kind == "graph" else int(2 ** rng.uniform(0, 5.5)),
            "levels_seed": rng.randrange(1 << 20)}
    if kind == "batch":
        case["shape"] = rng.choice(["default", "tuned_batch"])
    return case


# ---- inputs -------------------------------------------------------------------------------------------
_contexts = {}  # a program keeps its contexts: their tables depend on the parameters alone


def context(params):
    if params not in _contexts:
        logN, L, K, alpha, qb, pb, h = params
        _contexts[params] = he.Context(he.Params(logN, L, K, alpha, qb, pb, h), device=True)
    return _contexts[params]


def generator(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def residues(lead, moduli, N, gen):
    """[*lead][len(moduli)][N] uniform residues."""
    out = torch.empty((*lead, len(moduli), N), dtype=torch.int64, device=DEV)
    for i, m in enumerate(moduli):
        out[..., i, :] = torch.randint(0, int(m), (*lead, N), generator=gen, device=DEV)
    return out


def words(lead, bits, N, gen):
    """[*lead][ceil(bits / 64)][N] uniform little-endian integers below 2^bits."""
    n = (bits + 63) // 64
    out = torch.randint(-(1 << 63), (1 << 63) - 1, (*lead, n, N), generator=gen, device=DEV)
    if bits % 64:
        out[..., n - 1, :] &= (1 << (bits % 64)) - 1
    return out


def eval_key(ctx, gen):
    return residues((ctx.dnum, 2), ctx.moduli, ctx.N, gen)


def empty(*shape):
    return torch.empty(shape, dtype=torch.int64, device=DEV)


def make_jobs(ctx, levels, gen):
    return [(residues((2,), ctx.q[:lv], ctx.N, gen), residues((2,), ctx.q[:lv], ctx.N, gen),
             empty(2, lv - 1, ctx.N), lv) for lv in levels]


def set_shape(ctx, name):
    he.he_set_shape(ctx, *(SHAPES[name] or (4, 8, 1, 0, 8, 7, 0, 0, 0)))


def serve_requests(case):
    """(ring, level) per request: 70 % N = 2^15 at levels 2..16, 30 % N = 2^16 at levels 4..24."""
    g = np.random.Generator(np.random.PCG64(case["levels_seed"]))
    return [("n15", int(g.integers(2, 17))) if g.random() < 0.7 else ("n16", int(g.integers(4, 25)))
            for _ in range(case["jobs"])]


def prepare(case, seed):
    gen = generator(seed)
    st = {"case": case}
    kind = case["kind"]
    if kind == "bigint":
        logN, logQ, logq = case["logN"], case["logQ"], case["logq"]
        # primes of 57 bits, enough for products of 3 log Q bits
        ctx = context((logN, min(64, (3 * logQ + logN + 2) // 56 + 2), 1, 16, 57, 57, 64))
        plan = he.NrPlan(ctx, logQ, case["logp"])
        N = ctx.N
        st.update(ctx=ctx, plan=plan, a=words((2,), logq, N, gen), b=words((2,), logq, N, gen),
                  key=plan.prepare_evk(words((2,), 2 * logQ, N, gen)), ws=plan.workspace(),
                  out=empty(2, (logq + 63) // 64, N), rs=empty(2, (logq - case["logp"] + 63) // 64, N))
        return st
    if kind == "serve":
        ctxs = {r: context(RINGS[r]) for r in ("n15", "n16")}
        for c in ctxs.values():
            set_shape(c, "default")
        keys = {r: eval_key(c, gen) for r, c in ctxs.items()}
        jobs = []
        for ring, lv in serve_requests(case):
            (a, b, o, _), = make_jobs(ctxs[ring], [lv], gen)
            jobs.append((0 if ring == "n15" else 1, lv, a, b, o))
        server = he.Server([ctxs["n15"], ctxs["n16"]], [keys["n15"], keys["n16"]], 4 << 30, max_batch=64, streams=4)
        torch.cuda.synchronize()
        st.update(server=server, jobs=jobs, keys=keys)
        return st
    ctx = context(RINGS[case["ring"]])
    N = ctx.N
    set_shape(ctx, case.get("shape", "default"))
    st["ctx"] = ctx
    if kind == "single":
        lv, call = case["level"], case["call"]
        st.update(a=residues((2,), ctx.q[:lv], N, gen), b=residues((2,), ctx.q[:lv], N, gen),
                  ws=he.workspace(ctx, lv),
                  out=empty(2, lv if call in ("mul", "rotate") else lv - 1, N))
        if call == "mul_rescale_seeded":
            st["key"] = residues((ctx.dnum,), ctx.moduli, N, gen)
            he.he_evk_register_seeded(ctx, st["key"], seed)
            # the registration is by address: it ends with the key's memory
            weakref.finalize(st["key"], he.lib().he_evk_unregister, ctx.ptr, st["key"].data_ptr())
        else:
            st["key"] = eval_key(ctx, gen)
        if call == "rotate":
            st["galois"] = he.he_galois_elt(ctx, 5)
    elif kind == "linear":
        lv = case["level"]
        q = ctx.q[:lv]
        st.update(a=residues((2,), q, N, gen), b=residues((2,), q, N, gen), pa=residues((), q, N, gen),
                  pb=residues((), q, N, gen), wa=empty(2, lv, N), wb=empty(2, lv, N), out=empty(2, lv - 1, N),
                  ws=he.workspace(ctx, lv))
    else:
        levels = batch_levels(case["jobs"], case["levels_lo"], case["levels_hi"], case["levels_seed"])
        st["key"] = eval_key(ctx, gen)
        if kind == "host":
            host = [[torch.empty((2, n, N), dtype=torch.int64, pin_memory=True) for n in (lv, lv, lv - 1)]
                    for lv in levels]
            for bufs, lv in zip(host, levels):
                for k in range(2):
                    bufs[k].copy_(residues((2,), ctx.q[:lv], N, gen))
            st["host"], st["levels"] = host, levels
            st["in1"], st["in2"], st["outs"] = ([b[k].numpy().view(np.uint64) for b in host] for k in range(3))
            st["ws"] = empty(he.he_host_stream_workspace_bytes(ctx, max(levels), 2) // 8)
        else:
            st["jobs"] = make_jobs(ctx, levels, gen)
            if kind == "batch":
                st["ws"] = empty(he.he_batch_workspace_bytes(ctx, levels) // 8)
            else:
                st["graph"] = he.BatchGraph(ctx, case["jobs"], st["key"])
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "bigint":
        plan, logq = st["plan"], case["logq"]
        plan.mul(st["a"], st["b"], st["key"], logq, st["out"], st["ws"])
        plan.rescale(st["out"], logq, st["rs"])
        return [st["out"], st["rs"]]
    if kind == "serve":
        tickets = [st["server"].submit(*job) for job in st["jobs"]]
        for t in tickets:
            st["server"].wait(t)
        return [job[4] for job in st["jobs"]]
    ctx = st["ctx"]
    if kind == "single":
        lv, call = case["level"], case["call"]
        if call == "rotate":
            he.he_rotate(ctx, st["a"], st["key"], lv, st["galois"], st["out"], st["ws"])
        elif call == "mul":
            he.he_mul(ctx, st["a"], st["b"], st["key"], lv, st["out"], st["ws"])
        elif call == "mul_rescale_pq":
            he.he_mul_rescale_pq(ctx, st["a"], st["b"], st["key"], lv, st["out"], st["ws"])
        else:
            he.he_mul_rescale(ctx, st["a"], st["b"], st["key"], lv, st["out"], st["ws"])
        return st["out"]
    if kind == "linear":
        lv = case["level"]
        he.he_mul_plain(ctx, st["a"], st["pa"], lv, st["wa"])
        he.he_mul_plain(ctx, st["b"], st["pb"], lv, st["wb"])
        he.he_add(ctx, st["wa"], st["wb"], lv, st["wa"])
        he.he_rescale(ctx, st["wa"], lv, st["out"], st["ws"])
        return st["out"]
    if kind == "host":
        he.he_mul_rescale_host_stream(ctx, st["in1"], st["in2"], st["levels"], st["outs"], st["key"], st["ws"])
        return st["outs"]
    if kind == "batch":
        he.he_mul_batch(ctx, st["jobs"], st["key"], st["ws"])
    else:
        st["graph"].launch(st["jobs"])
    return [job[2] for job in st["jobs"]]


# ---- what a pass cannot do without ----------------------------------------------------------------------
def _mul_work(ring, level, call):
    """(bytes without the key, key bytes, word operations) of one key switch at `level`.  A butterfly or a
    modular multiply-add counts as two operations."""
    logN, L, K, alpha, _, _, _ = RINGS[ring]
    N = 1 << logN
    beta = -(-level // alpha)
    lout = level if call in ("mul", "rotate") else level - 1
    operands = (1 if call == "rotate" else 2) * 2 * level + 2 * lout
    key = beta * (1 if call == "mul_rescale_seeded" else 2) * (K + level)
    extra = 0 if lout == level else 2
    transforms = level + extra + beta * (K + level) - level + 2 * K + extra + 2 * lout
    macs = (beta * (K + level) - level) * alpha + 2 * level * K  # base conversions
    macs += 2 * beta * (K + level) + (0 if call == "rotate" else 4 * level) + 2 * level
    return operands * N * 8, key * N * 8, 2 * (transforms * N // 2 * logN + macs * N)


def work(case):
    kind = case["kind"]
    if kind == "bigint":
        N, wq = 1 << case["logN"], (case["logq"] + 63) // 64
        w2 = (2 * case["logQ"] + 63) // 64
        np1 = -(-(2 * case["logQ"] + case["logN"] + 2) // 57)
        np2 = -(-(3 * case["logQ"] + case["logN"] + 2) // 57)
        wo = (case["logq"] - case["logp"] + 63) // 64
        conv = N * (4 * wq * np1 + 3 * np1 * wq + wq * np2 + 2 * np2 * w2)  # word products of CRT and iCRT
        ntt = N // 2 * case["logN"] * (7 * np1 + 3 * np2)
        return {"bytes": 8 * N * (4 * wq + 2 * np2 + 2 * wq + 2 * wq + 2 * wo), "flops": 2 * (conv + ntt + N * (4 * np1 + 2 * np2))}
    if kind == "single":
        b, k, f = _mul_work(case["ring"], case["level"], case["call"])
        return {"bytes": b + k, "flops": f}
    if kind == "linear":
        logN, lv = RINGS[case["ring"]][0], case["level"]
        N = 1 << logN
        return {"bytes": 8 * N * (4 * lv + 2 * lv + 2 * (lv - 1)),
                "flops": 2 * (N * (6 * lv + 2 * lv) + 2 * lv * N // 2 * logN)}
    if kind == "serve":
        jobs = serve_requests(case)
    else:
        jobs = [(case["ring"], lv) for lv in batch_levels(case["jobs"], case["levels_lo"], case["levels_hi"],
                                                          case["levels_seed"])]
    parts = [(ring, *_mul_work(ring, lv, "mul_rescale")) for ring, lv in jobs]
    keys = {}
    for ring, _, k, _ in parts:  # one key serves every job of a ring
        keys[ring] = max(keys.get(ring, 0), k)
    return {"bytes": sum(p[1] for p in parts) + sum(keys.values()), "flops": sum(p[3] for p in parts)}


def exact(case, seed):
    """Every output is whole numbers, equal word for word in every build: nothing to compare in floating point."""
    return None
