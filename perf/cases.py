"""The decode work whose speed this repository is measured by, as a program that serves a model has it done.

One pass of a case is one window of one layer through the public calls of `binding.SketchSSM`:
- path "window": buf_len - 1 decode steps and the state update that ends the window (Algorithm 1 in lock step);
- path "mixed":  buf_len calls of the continuous-batching step, every sequence at a window phase of its own, so that
                 every call serves decode steps at all ring fills beside flushes;
- path "replay": the exact buffered replay (full-state-read decode steps, a state update without the sketch): what a
                 layer runs whose heads are not sketched.
With `admit` the pass begins by building the sketch (and the map) from a state that a prefill left.
After a pass every sequence is at the window phase where it began, so passes follow one another like windows do.

A case's values: kind, batch, heads, dk, dv, rank, buf_len (the layer), io (precision of q, k, v and of the ring), out
(precision of the outputs), sketch (storage of the sketch and of the map), coef ("fixed": the offline map; "pivot": the
state-dependent map with four pivots; "ridge": its exact form), erase (the coefficients through projected erase
vectors), ranks (a per-head rank table with a dense-fallback head), path, admit.
"""
import math

import torch

from paper_2609_33051_b200 import binding, traffic

_BASE = dict(path="window", kind="mamba2", batch=256, heads=64, dk=128, dv=64, rank=16, buf_len=16, io="bf16", out="f32",
             sketch="f32", coef="fixed", erase=False, ranks=False, admit=False)


def _case(name, **kw):
    return dict(_BASE, name=name, **kw)


def listed():
    return [
        # the smallest layer: a tiny model or a single user, where the launches and their latency are the time
        _case("gdn_tiny_f32", kind="gdn", batch=4, heads=4, dk=64, dv=64, rank=8, buf_len=8, io="f32"),
        # the small end of the batch sweep: short kernels in a row
        _case("mamba2_small", batch=64, rank=8, buf_len=4),
        # the three layer workloads, one for each recurrence
        _case("mamba2_layer"),
        _case("gdn_layer", kind="gdn", batch=512, heads=32, dv=128),
        _case("kda_layer", kind="kda", batch=512, heads=32, dv=128, buf_len=32),
        # long windows and a large rank: ring reads and the replay of 64 tokens weigh most
        _case("mamba2_long", rank=32, buf_len=64),
        # a layer of the large-batch stack: the largest call, bound by memory
        _case("mamba2_stack", batch=2048),
        # the paper's own configuration: state-dependent map, bfloat16 sketch and map
        _case("mamba2_statedep_bf16", coef="pivot", sketch="bf16"),
        # the same for the delta rule, with the projected erase vectors
        _case("gdn_statedep_erase", kind="gdn", batch=512, heads=32, dv=128, coef="pivot", sketch="bf16", erase=True),
        # continuous batching: sequences join at different times, every call mixes decode steps and flushes
        _case("gdn_mixed", kind="gdn", path="mixed", batch=512, heads=32, dv=128),
        # odd sizes: 80 value channels, a rank that is no multiple of four, ranks per head with a dense head, an odd batch,
        # admission of the batch from a prefilled state first, bfloat16 outputs
        _case("mamba2_v80_ragged", batch=37, heads=24, dv=80, rank=13, buf_len=12, ranks=True, admit=True, out="bf16"),
        # exact replay with 32-bit inputs: reads the whole state every step
        _case("kda_f32_replay", kind="kda", path="replay", batch=96, heads=32, dv=128, buf_len=8, io="f32"),
    ]


_MOST_BYTES = 8e9       # of the state alone, below the largest listed case in memory, bytes moved and time


def draw(rng):
    """One more case of the ranges that the listed ones stand for."""
    while True:
        c = dict(_BASE)
        c["path"] = rng.choice(["window"] * 6 + ["mixed", "replay"])
        c["kind"] = rng.choice(["mamba2", "gdn", "kda"])
        c["dk"], c["dv"] = rng.choice([(128, 64), (128, 64), (128, 128), (128, 128), (128, 128), (128, 80), (64, 64)])
        c["batch"] = round(math.exp(rng.uniform(math.log(1), math.log(2048))))
        c["heads"] = rng.choice([4, 8, 16, 24, 32, 32, 48, 64])
        c["rank"] = rng.choice([8, 8, 13, 16, 16, 16, 24, 32])
        c["buf_len"] = rng.choice([4, 8, 12, 16, 16, 16, 20, 32, 32, 64])
        c["io"] = rng.choice(["bf16"] * 5 + ["f32"])
        c["out"] = rng.choice(["f32", "f32", "bf16"])
        if c["path"] != "replay":
            c["sketch"] = rng.choice(["f32", "f32", "bf16"])
            c["coef"] = rng.choice(["fixed", "fixed", "fixed", "pivot", "pivot", "ridge"])
            c["ranks"] = c["coef"] == "fixed" and rng.random() < 0.2
            c["admit"] = c["path"] == "window" and rng.random() < 0.2
            c["erase"] = (c["kind"] != "mamba2" and c["path"] == "window" and c["buf_len"] <= 32 and c["rank"] % 8 == 0 and
                          rng.random() < 0.25)
        if work(c)["bytes"] <= _MOST_BYTES and c["batch"] * c["heads"] >= 4:
            return c


# ---- what a program has in hand ---------------------------------------------------------------------------------------

_TORCH = {"f32": torch.float32, "bf16": torch.bfloat16}


def _tokens(c, steps, gen):
    """Token tensors of `steps` decode steps, [steps, B, H, ...] on the device, rounded to the I/O precision."""
    B, H, K, V = c["batch"], c["heads"], c["dk"], c["dv"]
    io = _TORCH[c["io"]]

    def normal(*shape):
        return torch.randn(steps, B, H, *shape, device="cuda", generator=gen)

    q, k, v, zb = normal(K), normal(K), normal(V), normal()
    if c["kind"] == "mamba2":
        beta = torch.nn.functional.softplus(zb)                               # the step size
        a_log = 2.7 * torch.rand(H, device="cuda", generator=gen)
        decay = torch.exp(-beta * torch.exp(a_log))
    else:
        q = q / q.norm(dim=-1, keepdim=True)
        k = k / k.norm(dim=-1, keepdim=True)
        beta = torch.sigmoid(zb).to(io).float()
        if c["kind"] == "gdn":
            decay = torch.exp(-torch.nn.functional.softplus(normal()))
        else:
            decay = torch.sigmoid(2.0 + normal(K)).to(io)
    return dict(q=q.to(io), k=k.to(io), v=v.to(io), beta=beta.contiguous(), decay=decay.contiguous())


def _basis(c, seed):
    """Orthonormal sketching matrices [H, K, r], one per head, and the offline map that goes with them (the transpose)."""
    gen = torch.Generator().manual_seed(seed)
    om = torch.linalg.qr(torch.randn(c["heads"], c["dk"], c["rank"], dtype=torch.float64, generator=gen))[0].float()
    return om, om.transpose(1, 2).contiguous()


def _rank_table(c):
    """Ranks as an offline allocation gives them: full, half and small ranks and one dense-fallback head."""
    r = c["rank"]
    return [[r, r, max(1, r // 2), r, max(1, r // 4), 0][h % 6] if h < 12 or h % 6 != 5 else r for h in range(c["heads"])]


def _phases(c, seed):
    """Ring fill of every sequence at the start of a pass."""
    if c["path"] != "mixed":
        return torch.zeros(c["batch"], dtype=torch.int64)
    return torch.randint(0, c["buf_len"], (c["batch"],), generator=torch.Generator().manual_seed(seed))


def _inputs(c, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    state = torch.randn(c["batch"], c["heads"], c["dk"], c["dv"], device="cuda", generator=gen) * 0.02
    tokens = _tokens(c, c["buf_len"], gen)
    held = _tokens(c, c["buf_len"], gen) if c["path"] == "mixed" else None     # what the ring already holds
    omega, coef = _basis(c, seed)
    return state, tokens, held, omega, coef, _phases(c, seed)


def prepare(case, seed):
    c = dict(_BASE, **case)
    state, tokens, held, omega, coef, fill = _inputs(c, seed)
    m = binding.SketchSSM(c["kind"], c["batch"], c["heads"], c["dk"], c["dv"], c["rank"], c["buf_len"], io=c["io"], out=c["out"],
                          coef_per_seq=c["coef"] != "fixed", coef_pivots=0 if c["coef"] == "ridge" else 4,
                          sketch=c["sketch"], erase_factors=c["erase"])
    m.state.copy_(state)
    del state
    m.omega.copy_(omega)
    if c["coef"] == "fixed":
        m.coef.copy_(coef)
    if c["ranks"]:
        m.head_rank = torch.tensor(_rank_table(c), dtype=torch.int32, device="cuda")
    m.bind()
    if c["path"] != "replay" and not c["admit"]:
        m.state_update(0)                                                      # the sketch of the prefilled state
    if held is not None:
        for view, name in zip(m.ring_views(), ("k", "v", "beta", "decay")):
            view.copy_(held[name].movedim(0, 2))
        m.bind()
    L = c["buf_len"]
    out = torch.empty(L, c["batch"], c["heads"], c["dv"], dtype=_TORCH[c["out"]], device="cuda")
    s = dict(path=c["path"], admit=c["admit"], layer=m, out=out, last=L - 1,
             steps=[tuple(tokens[n][t] for n in ("q", "k", "v", "beta", "decay")) + (out[t],) for t in range(L)])
    if c["path"] == "mixed":
        now = (fill[None, :] + torch.arange(L)[:, None]) % L
        s["phase"] = list(torch.where(now == L - 1, -L, now).to(torch.int32).cuda())
    return s


def run(s):
    m = s["layer"]
    if s["path"] == "mixed":
        for phase, step in zip(s["phase"], s["steps"]):
            m.step_mixed(phase, *step)
        return dict(out=s["out"], state=m.state, sketch=m.sketch, coef=m.coef if m.coef_per_seq else None, ring=m.ring)
    if s["path"] == "replay":
        for n in range(s["last"]):
            m.full_read_decode(n, *s["steps"][n])
        m.state_update(s["last"], *s["steps"][s["last"]], flags=binding.NO_SKETCH)
        return dict(out=s["out"], state=m.state)
    if s["admit"]:
        m.state_update(0)
    for n in range(s["last"]):
        m.decode_step(n, *s["steps"][n])
    m.state_update(s["last"], *s["steps"][s["last"]])
    return dict(out=s["out"], state=m.state, sketch=m.sketch, coef=m.coef if m.coef_per_seq else None)


# ---- what a pass cannot do without -------------------------------------------------------------------------------------

def work(case):
    c = dict(_BASE, **case)
    kind, B, H, K, V, r, L, io = (c[n] for n in ("kind", "batch", "heads", "dk", "dv", "rank", "buf_len", "io"))
    full = c["path"] == "replay"
    kw = dict(io=io, out_bytes=2 if c["out"] == "bf16" else 4, sketch_bytes=2 if c["sketch"] == "bf16" else 4,
              coef_per_seq=c["coef"] != "fixed")
    total = sum(traffic.decode_bytes(kind, B, H, K, V, r, n, full_read=full, erase_factors=c["erase"], **kw) for n in range(L - 1))
    total += traffic.update_bytes(kind, B, H, K, V, r, L - 1, sketch=not full, **kw)
    flops = 0
    for n in range(L - 1):                                                     # sweep, map, rows, buffered values
        flops += 4 * K * (n + 1) + 2 * V * (n + 1) + (2 * K * V if full else 2 * r * (K + V))
    flops += 2 * L * K * V * (1 if kind == "mamba2" else 2) + 2 * K * V * (1 if full else r + 1)
    if c["admit"]:
        total += B * H * (K * V * 4 + r * V * kw["sketch_bytes"])
        flops += 2 * K * V * r
    return {"bytes": total, "flops": flops * B * H}


def tolerance(case):
    """About four times the distance from the 64-bit results that was measured: 5e-4 where the sketch and the map are
    stored in bfloat16 (an element beside a rounding boundary moves the map), 2e-5 with 16-bit inputs (their products
    with operands split in two bfloat16 halves), 2e-6 with 32-bit inputs (the maps' linear systems among them); outputs
    in bfloat16 differ by single roundings."""
    c = dict(_BASE, **case)
    if "bf16" in (c["sketch"], c["out"]):
        return {"rel": 2e-3}
    return {"rel": 1e-4 if c["io"] == "bf16" else 1e-5}


# ---- the same in 64 bits ------------------------------------------------------------------------------------------------

def _maps(c, S, U, omega):
    """State-dependent maps [b, H, r, K] of S [b, H, K, V] and the stored sketch U [b, H, r, V] (ridge 0.1)."""
    lam, p = 0.1, min(c["rank"], 4)
    mu = S.square().sum((-1, -2)) / S.shape[-2]
    mu = torch.where(mu == 0, torch.ones_like(mu), mu)[..., None, None]
    if c["coef"] == "ridge":
        eye = torch.eye(c["rank"], dtype=S.dtype, device=S.device)
        return torch.linalg.solve(U @ U.mT + lam * mu * eye, U @ S.mT)
    Q = torch.linalg.qr(U[..., :p, :].mT)[0]                                   # an orthonormal basis of the first p columns
    LG = U @ Q / mu.sqrt()
    d = ((U.square().sum(-1) - (U @ Q).square().sum(-1)) / mu[..., 0]).clamp_min(0)[..., None]
    rhs = (LG @ (Q.mT @ S.mT) / mu.sqrt() + d * omega.mT) / (d + lam)
    F = LG / (d + lam)
    TP = torch.eye(p, dtype=S.dtype, device=S.device) + LG.mT @ F
    return rhs - F @ torch.linalg.solve(TP, LG.mT @ rhs)


def _exact_part(c, state, tokens, held, omega, coef, fill):
    """out [L, b, H, V], state, sketch, coef of one pass over a part of the batch; everything in 64 bits but the stored
    sketch and map, which have the precision that their storage has."""
    L, kind, r = c["buf_len"], c["kind"], c["rank"]
    f64 = torch.float64
    S = state.to(f64)
    b, H, K, V = S.shape
    om, ranks = omega.to(S), torch.tensor(_rank_table(c) if c["ranks"] else [r] * c["heads"], device=S.device)

    def stored(x):
        return x.float().bfloat16().to(f64) if c["sketch"] == "bf16" else x

    def sketch_of(S):
        U = stored(om.mT @ S)
        return U, (stored(_maps(c, S, U, om)) if c["coef"] != "fixed" else C)

    live = torch.arange(r, device=S.device)[None, :, None] < ranks[:, None, None]
    C = stored(coef.to(S)) * live
    dense = (ranks == 0)[:, None]
    if c["path"] != "replay":
        U, C = sketch_of(S)
    ring = {n: [held[n][t].to(f64) for t in range(L)] if held is not None else [None] * L for n in ("k", "v", "beta", "decay")}
    n_now = fill.to(S.device)
    outs = []
    for t in range(L):
        q = tokens["q"][t].to(f64)
        lock = held is None
        for name in ring:
            new = tokens[name][t].to(f64)
            if lock:
                ring[name][t] = new
            else:
                for s in range(L):
                    at = (n_now == s).view(b, *([1] * (new.dim() - 1)))
                    ring[name][s] = torch.where(at, new, ring[name][s])

        def gate(s):
            g = ring["decay"][s]
            return g if kind == "kda" else g[..., None]

        slots = range(t + 1) if lock else range(L)
        x, o = q.clone(), torch.zeros(b, H, V, dtype=f64, device=S.device)
        for s in reversed(slots):                                              # effective query and buffer output
            there = (n_now >= s)[:, None, None] if not lock else None
            a = ring["beta"][s][..., None] * (ring["k"][s] * x).sum(-1, keepdim=True)
            y = gate(s) * (x - a * ring["k"][s] if kind != "mamba2" else x)
            if lock:
                x, o = y, o + a * ring["v"][s]
            else:
                x, o = torch.where(there, y, x), o + torch.where(there, a * ring["v"][s], torch.zeros_like(o))
        exact = (S.mT @ x[..., None])[..., 0]
        if c["path"] == "replay":
            o = o + exact
        else:
            read = (U.mT @ (C @ x[..., None]))[..., 0]
            o = o + torch.where(dense, exact, read)
        flush = n_now == L - 1
        if bool(flush.any()):
            f = flush.nonzero()[:, 0]
            Sf = S[f]
            for s in range(L):
                k, v, beta = ring["k"][s][f][..., None], ring["v"][s][f][..., None, :], ring["beta"][s][f][..., None, None]
                Sf = gate(s)[f][..., None] * Sf
                Sf = Sf + beta * k * (v - k.mT @ Sf if kind != "mamba2" else v)
            S[f] = Sf
            o[f] = (Sf.mT @ q[f][..., None])[..., 0]
            if c["path"] != "replay":
                Uf, Cf = sketch_of(Sf)
                U[f] = Uf
                if c["coef"] != "fixed":
                    C[f] = Cf
        n_now = (n_now + 1) % L
        outs.append(o)
    got = dict(out=torch.stack(outs), state=S)
    if c["path"] != "replay":
        got.update(sketch=U)
    if c["coef"] != "fixed":
        got.update(coef=C)
    return got


def exact(case, seed):
    c = dict(_BASE, **case)
    state, tokens, held, omega, coef, fill = _inputs(c, seed)
    omega, coef = omega.cuda(), coef.cuda()
    per = max(1, (1 << 27) // (c["heads"] * c["dk"] * c["dv"]))
    parts = []
    for b in range(0, c["batch"], per):
        cut = {n: x[:, b:b + per] for n, x in tokens.items()}
        old = {n: x[:, b:b + per] for n, x in held.items()} if held is not None else None
        parts.append(_exact_part(c, state[b:b + per], cut, old, omega, coef, fill[b:b + per]))
    got = {n: torch.cat([p[n] for p in parts], dim=1 if n == "out" else 0) for n in parts[0]}
    if c["path"] == "replay":
        return got
    got.setdefault("coef", None)
    if c["path"] == "mixed":
        got["ring"] = None                                                     # bytes: no value in 64 bits
    return got
