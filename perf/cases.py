"""Performance cases of the RhymeFlow step core: what a user's program has it do.

``listed()`` gives the named cases and ``draw(rng)`` more of the same ranges; ``prepare`` makes
the inputs and handles that a program holds before the call, ``run`` makes one pass through the
public entry points, ``work`` states the bytes and operations a pass cannot do without,
``tolerance`` how far another correct implementation may be off, and ``exact`` the result in 64
bits from plain torch.

Kinds of case:
  step      one asynchronous denoising step, ``StepCore.run`` (compaction, latent projection,
            K/V-cache projection, attention, Euler update)
  graph     a whole trajectory recorded by ``StepCore.capture_trajectory`` and replayed
  attn      the attention of one layer, ``rf_attn`` / ``rf_attn_noalloc``
  masked    the attention of one layer under a token block mask, ``rf_attn_block_masked``
  kv        one layer's rolling K/V cache, ``rf_project_kv``
  gram      similarities of the clean-latent proxies, ``rf_frame_gram`` (keyframe selection)
  pipeline  a short trajectory fed from pinned host memory, ``HostPipeline``

Shapes: F latent frames of N tokens, H heads of dim d, C latent channels per token, S steps, a
keyframe every ``gap`` frames (and the last frame), non-keyframes skipping ``stride`` steps.
"""
import math

import torch

import paper_2606_06309_gb300 as rf
from paper_2606_06309_gb300.stepcore import HostPipeline, StepCore, upload_plan

DEV = "cuda"
# exact() computes attention up to this many operations (64-bit rates: some seconds)
EXACT_FLOPS = 3.0e12


# ------------------------------------------------------------------------------ the cases
def listed():
    return [
        # The smallest step: 4 frames of 8 x 8 tokens, head dim 64, only the keyframes active.
        # Five short launches: latency and host work count.
        dict(name="step_tiny", kind="step", F=4, N=64, H=2, d=64, C=16, S=4, gap=3, stride=2, s=1),
        # The same video's whole trajectory as one CUDA graph: what a program that denoises
        # many small videos replays.
        dict(name="graph_tiny", kind="graph", F=4, N=64, H=2, d=64, C=16, S=4, gap=3, stride=2),
        # A keyframe-only step of a short 480p clip: few rows against all keys, the projection
        # of nine frames' keys and values in front of it.
        dict(name="step_480p_keys", kind="step", F=13, N=1560, H=12, d=128, C=16, S=20, gap=4,
             stride=2, s=1),
        # A step of the usual 81-frame 480p clip with every frame active.
        dict(name="step_480p_all", kind="step", F=21, N=1560, H=12, d=128, C=16, S=50, gap=5,
             stride=4, s=0),
        # The largest: every frame of a long 720p video active, 118800 tokens.
        dict(name="step_720p_long_all", kind="step", F=33, N=3600, H=24, d=128, C=16, S=50,
             gap=7, stride=6, s=0),
        # Head dim 64 (the models with many narrow heads), attention alone.
        dict(name="attn_d64", kind="attn", F=13, N=1560, H=24, d=64, A=13, layout="packed",
             scratch="workspace", lse=False),
        # Odd sizes: tiles across frames, a ragged last key tile, rows of a fused QKV buffer,
        # log-sum-exps kept, and the library's own scratch.
        dict(name="attn_ragged_fused", kind="attn", F=7, N=1003, H=5, d=128, A=5,
             layout="fused", scratch="noalloc", lse=True),
        # Combined frame and token mask, keyframe-only step: few short items.
        dict(name="masked_480p_keys", kind="masked", F=13, N=1560, H=12, d=128, A=4,
             pattern="band", density=0.23),
        # Combined mask on a 720p clip with 40 heads, every frame active.
        dict(name="masked_720p_all", kind="masked", F=21, N=3600, H=40, d=128, A=21,
             pattern="band", density=0.23),
        # One layer's cache step of a keyframe-only step of the long 720p video.
        dict(name="kv_720p_long_keys", kind="kv", F=33, N=3600, H=24, d=128, A=6,
             layout="packed"),
        # Keyframe selection of the long video over its latent proxies.
        dict(name="gram_latent", kind="gram", F=33, E=57600),
        # Tensors that live in host memory: four steps of a short clip, copies included.
        dict(name="pipeline_480p", kind="pipeline", F=13, N=1560, H=12, d=128, C=16, S=4, gap=4,
             stride=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["step", "graph", "attn", "masked", "kv", "gram", "pipeline"],
                       [5, 1, 4, 3, 2, 2, 1])[0]
    if kind == "gram":  # latent width up to the width of a layer's hidden state
        F = rng.randint(1, 64)
        return dict(kind="gram", F=F, E=_log_int(rng, 1000, min(11_000_000, 400_000_000 // F)))
    while True:
        F = _log_int(rng, 2, 33)
        N = _log_int(rng, 16, 3600)
        H = _log_int(rng, 1, 40)
        d = rng.choice([64, 128, 128])
        most = {"graph": 2e11, "pipeline": 2e12}.get(kind, 1.2e14)
        # a size is taken if the work is bounded, and tiny ones are not drawn most of the time
        if 4.0 * (F * N) ** 2 * H * d <= most and F * N * H * d <= 3.0e8 and F * N >= 64:
            break
    c = dict(kind=kind, F=F, N=N, H=H, d=d)
    if kind in ("step", "graph", "pipeline"):
        S = rng.randint(2, 6)
        c.update(C=rng.choice([4, 16, 16, 64]), S=S, gap=rng.randint(2, 8),
                 stride=rng.randint(1, 4))
        if kind == "step":
            c["s"] = rng.randrange(S)
    else:
        c["A"] = rng.randint(1, F)
    if kind in ("attn", "kv"):
        c["layout"] = rng.choice(["packed", "packed", "fused"])
    if kind == "attn":
        c.update(scratch=rng.choice(["workspace", "workspace", "noalloc", "none"]),
                 lse=rng.random() < 0.5)
    if kind == "masked":
        c.update(pattern=rng.choice(["band", "causal", "random"]),
                 density=round(rng.uniform(0.1, 0.9), 3))
    return c


# ------------------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed & 0x7FFFFFFFFFFF)


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float32)


def _bf16(g, *shape):
    return _normal(g, *shape).to(torch.bfloat16)


def _keys(c):
    F = c["F"]
    return [1 if f % c["gap"] == 0 or f == F - 1 else 0 for f in range(F)]


def _active_mask(F, A):
    m = [0] * F
    for i in range(A):
        m[i * F // A] = 1
    return m


def _block_mask(c, g):
    """uint8 [H][nb][nb] over blocks of 128 tokens."""
    nb = -(-c["F"] * c["N"] // 128)
    i = torch.arange(nb, device=DEV)
    dist = (i[:, None] - i[None, :]).abs()
    if c["pattern"] == "band":  # |qb - kb| <= w covers about `density` of the blocks
        w = int(nb * (1.0 - math.sqrt(max(0.0, 1.0 - c["density"]))))
        one = (dist <= w)
        m = one[None].expand(c["H"], nb, nb)
    elif c["pattern"] == "causal":
        m = (i[:, None] >= i[None, :])[None].expand(c["H"], nb, nb)
    else:  # scattered blocks, another set per head, the diagonal always kept
        m = torch.rand(c["H"], nb, nb, generator=g, device=DEV) < c["density"]
        m = m | (dist == 0)[None]
    return m.to(torch.uint8).contiguous()


def _qkv(c, g, layout="packed"):
    """bf16 Q, K, V [F*N, H, d]: three buffers, or slices of one fused [F*N, 3, H, d] buffer."""
    S_tok, H, d = c["F"] * c["N"], c["H"], c["d"]
    if layout == "fused":
        b = _bf16(g, S_tok, 3, H, d)
        return b[:, 0], b[:, 1], b[:, 2]
    return tuple(_bf16(g, S_tok, H, d) for _ in range(3))


def _lists(c):
    """Active / skipped lists and counts on the device, as rf_schedule_compact writes them."""
    F = c["F"]
    mask = torch.tensor(_active_mask(F, c["A"]), dtype=torch.uint8, device=DEV)
    act, skp = (torch.zeros(F, dtype=torch.int32, device=DEV) for _ in range(2))
    cnt = torch.zeros(2, dtype=torch.int32, device=DEV)
    rf.rf_schedule_compact(mask, F, c["N"], act, skp, None, cnt)
    return act, skp, cnt


def _workspace(d):
    n = rf.rf_attn_workspace_bytes(d)
    return torch.zeros((n + 3) // 4, dtype=torch.int32, device=DEV)


def _plan(c):
    return upload_plan(c["F"], c["S"], _keys(c), [c["stride"]] * c["S"], 0, DEV)


def _inputs(c, seed):
    """The random inputs of a case by name; prepare() and exact() both start from these."""
    g = _gen(seed * 1009 + 17)
    kind, t = c["kind"], {}
    if kind == "gram":
        # a video of a few scenes: frames of one scene share most of their content
        F, E = c["F"], c["E"]
        scenes = _normal(g, 4, E)
        t["P"] = _normal(g, F, E).mul_(0.4).add_(scenes[torch.arange(F, device=DEV) * 4 // F])
        return t
    F, N, D = c["F"], c["N"], c["H"] * c["d"]
    if kind in ("step", "graph", "pipeline"):
        E, S = N * c["C"], c["S"]
        t["z"] = _normal(g, 2, F, E)
        t["v"] = [_normal(g, F, E) for _ in range(1 if kind == "step" else S)]
        t["Q"], t["K"], t["V"] = _qkv(c, g)
        if kind == "pipeline":  # fresh queries, keys and values alternate between two sets
            t["Q2"], t["K2"], t["V2"] = _qkv(c, g)
        # cached keys and values: both slots for a single step, the initial ones otherwise
        n = 2 if kind == "step" else 1
        t["Kc"], t["Vc"] = _bf16(g, n, F, N, D), _bf16(g, n, F, N, D)
        return t
    t["Q"], t["K"], t["V"] = _qkv(c, g, c.get("layout", "packed"))
    if kind == "kv":
        t["Kc"], t["Vc"] = _bf16(g, 2, F, N, D), _bf16(g, 2, F, N, D)
        t["alpha"] = torch.rand(F, generator=g, device=DEV)
    if kind == "masked":
        t["mask"] = _block_mask(c, g)
    return t


def prepare(c, seed):
    t = _inputs(c, seed)
    kind = c["kind"]
    st = {"c": c, "t": t}
    if kind == "gram":
        st["G"] = torch.zeros(c["F"], c["F"], dtype=torch.float64, device=DEV)
        return st
    F, N, H, d = c["F"], c["N"], c["H"], c["d"]
    st["scale"] = 1.0 / math.sqrt(d)
    if kind in ("step", "graph", "pipeline"):
        plan = _plan(c)
        if kind == "pipeline":
            core = StepCore(F, N, N * c["C"], H, d, plan, DEV, kv_cache=False, split_kv=False)
            core.z2.copy_(t["z"])
            host = {k: t[k].cpu().pin_memory() for k in ("Q", "K", "V", "Q2", "K2", "V2")}
            host["v"] = [v.cpu().pin_memory() for v in t["v"]]
            host["O"] = torch.zeros(F * N, H, d, dtype=torch.bfloat16).pin_memory()
            host["z"] = torch.zeros(2, F, N * c["C"]).pin_memory()
            host["ctx"] = torch.zeros(F, N * c["C"]).pin_memory()
            st.update(pipe=HostPipeline(core, F * N, t["Kc"][0].cpu(), t["Vc"][0].cpu(), DEV),
                      host=host)
            for k in ("Q", "K", "V", "Q2", "K2", "V2", "Kc", "Vc", "v", "z"):
                del t[k]
            return st
        core = StepCore(F, N, N * c["C"], H, d, plan, DEV)
        st["core"] = core
        st["O"] = torch.zeros(F * N, H, d, dtype=torch.bfloat16, device=DEV)
        if kind == "step":
            core.z2.copy_(t.pop("z"))
            core.Kc.copy_(t.pop("Kc"))
            core.Vc.copy_(t.pop("Vc"))
        else:
            # the replay works on buffers of its own; each pass gives them the video's state
            core.set_state(t["z"][0])
            core.set_kv_cache(t["Kc"][0], t["Vc"][0])
            st["K"], st["V"] = t["K"].clone(), t["V"].clone()
            st["g"] = core.capture_trajectory(t["v"], st["O"], t["Q"], st["K"], st["V"],
                                              st["scale"])
        return st
    st["act"], st["skp"], st["cnt"] = _lists(c)
    if kind == "kv":
        st["beta"] = 1.0 - t["alpha"]
        st["slot"] = (torch.arange(F, device=DEV) % 2).to(torch.uint8)
        return st
    st["O"] = torch.zeros(F * N, H, d, dtype=torch.bfloat16, device=DEV)
    st["lse"] = (torch.zeros(H, F * N, device=DEV) if c.get("lse") or kind == "masked" else None)
    st["ws"] = (_workspace(d) if kind == "masked" or c["scratch"] == "workspace" else None)
    st["status"] = torch.zeros(1, dtype=torch.int32, device=DEV)
    return st


# ------------------------------------------------------------------------------ one pass
def run(st):
    c, t, kind = st["c"], st["t"], st["c"]["kind"]
    if kind == "gram":
        rf.rf_frame_gram(t["P"], st["G"])
        return {"G": st["G"]}
    F, N, H, d = c["F"], c["N"], c["H"], c["d"]
    if kind == "step":
        core = st["core"]
        core.run(c["s"], t["v"][0], st["O"], t["Q"], t["K"], t["V"], st["scale"])
        return {"O": st["O"], "ctx": core.ctx, "z": core.z2, "K": t["K"], "V": t["V"],
                "Kc": core.Kc, "Vc": core.Vc, "active": core.active, "skipped": core.skipped,
                "tokens": core.token_idx, "counts": core.counts, "status": core.status}
    if kind == "graph":
        core = st["core"]
        core.set_state(t["z"][0])
        core.set_kv_cache(t["Kc"][0], t["Vc"][0])
        st["K"].copy_(t["K"])
        st["V"].copy_(t["V"])
        st["g"].replay()
        return {"O": st["O"], "ctx": core.ctx, "z": core.z2, "K": st["K"], "V": st["V"],
                "Kc": core.Kc, "Vc": core.Vc, "status": core.status}
    if kind == "pipeline":
        h, p = st["host"], st["pipe"]
        for s in range(c["S"]):
            q, k, v = ("Q", "K", "V") if s % 2 == 0 else ("Q2", "K2", "V2")
            p.step(s, h[q], h[k], h[v], h["v"][s], h["O"], h["z"], st["scale"], h["ctx"])
        return {"O": h["O"], "z": h["z"], "ctx": h["ctx"], "status": p.sync()}
    if kind == "kv":
        K, V = t["K"], t["V"]
        rf.rf_project_kv(K, V, K.stride(0), t["Kc"], t["Vc"], st["slot"], t["alpha"], st["beta"],
                         st["act"], st["skp"], st["cnt"], F, N, H * d)
        return {"K": K, "V": V, "Kc": t["Kc"], "Vc": t["Vc"]}
    Q, K, V, O = t["Q"], t["K"], t["V"], st["O"]
    if kind == "masked":
        rf.rf_attn_block_masked(O, st["lse"], Q, K, V, Q.stride(0), O.stride(0), F, N, H, d,
                                st["act"], st["cnt"], st["scale"], t["mask"], st["ws"],
                                st["status"])
    elif c["scratch"] == "noalloc":
        rf.rf_attn_noalloc(O, st["lse"], Q, K, V, Q.stride(0), O.stride(0), F, N, H, d,
                           st["act"], st["cnt"], st["scale"], st["status"])
    else:
        rf.rf_attn(O, st["lse"], Q, K, V, Q.stride(0), O.stride(0), F, N, H, d, st["act"],
                   st["cnt"], st["scale"], st["ws"], st["status"])
    out = {"O": O, "status": st["status"]}
    if st["lse"] is not None:
        out["lse"] = st["lse"]
    return out


# ------------------------------------------------------------------------------ its work
def _schedule(c):
    """Algorithm 2 with the due-step rule: per step and frame (active, alpha, dt, slot)."""
    F, S, key = c["F"], c["S"], _keys(c)
    sig = [1.0 - s / S for s in range(S)] + [0.0]
    due, start, slot, rows = [0] * F, [0] * F, [0] * F, []
    for s in range(S):
        row = []
        for f in range(F):
            if key[f] or due[f] == s:
                nxt = min(s + (1 if key[f] else c["stride"]), S)
                row.append((1, 1.0, sig[nxt] - sig[s], slot[f]))
                start[f], due[f] = s, nxt
                slot[f] ^= 1
            else:
                a, b = sig[start[f]], sig[due[f]]
                row.append((0, (a - sig[s]) / (a - b), 0.0, slot[f]))
        rows.append(row)
    return rows


def _allowed_pairs(c):
    """(query, key) pairs of one head that a masked call cannot skip."""
    F, N = c["F"], c["N"]
    S_tok = F * N
    nb = -(-S_tok // 128)
    keys = [min(128, S_tok - 128 * b) for b in range(nb)]
    if c["pattern"] == "band":
        w = int(nb * (1.0 - math.sqrt(max(0.0, 1.0 - c["density"]))))
        span = [(max(0, b - w), min(nb, b + w + 1)) for b in range(nb)]
    elif c["pattern"] == "causal":
        span = [(0, b + 1) for b in range(nb)]
    else:
        span = None
    total = 0.0
    for f, on in enumerate(_active_mask(F, c["A"])):
        if not on:
            continue
        for b in range(f * N // 128, (f * N + N - 1) // 128 + 1):
            rows = min(f * N + N, 128 * b + 128) - max(f * N, 128 * b)
            if span is None:
                total += rows * (keys[b] + c["density"] * (S_tok - keys[b]))
            else:
                total += rows * sum(keys[span[b][0]:span[b][1]])
    return total


def _step_work(c, row):
    """One step: every input that has to be read once, every output written once."""
    F, N, H, d, E = c["F"], c["N"], c["H"], c["d"], c["N"] * c["C"]
    A = sum(r[0] for r in row)
    rows, S_tok, D = A * N, F * N, H * d
    latent = 4.0 * E * (2 * A + 3 * (F - A)) + 4.0 * E * 3 * A
    # K/V: active rows read and cached, skipped rows projected from two cached states; the
    # attention needs them once more only on chip
    kv = 2 * 2.0 * N * D * (2 * A + 3 * (F - A))
    return {"bytes": latent + kv + 2 * 2.0 * rows * D + 4.0 * rows,
            "flops": 4.0 * rows * S_tok * D}


def work(c):
    kind = c["kind"]
    if kind == "gram":
        F, E = c["F"], c["E"]
        return {"bytes": 4.0 * F * E + 8.0 * F * F, "flops": 1.0 * F * (F + 1) * E}
    if kind == "step":
        return _step_work(c, _schedule(c)[c["s"]])
    if kind in ("graph", "pipeline"):
        w = [_step_work(c, row) for row in _schedule(c)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    F, N, H, d, A = c["F"], c["N"], c["H"], c["d"], c["A"]
    D, S_tok = H * d, F * N
    if kind == "kv":
        return {"bytes": 2 * 2.0 * N * D * (2 * A + 3 * (F - A)), "flops": 2 * 3.0 * N * D * (F - A)}
    pairs = _allowed_pairs(c) if kind == "masked" else 1.0 * A * N * S_tok
    mask = H * (-(-S_tok // 128)) ** 2 if kind == "masked" else 0
    lse = 4.0 * H * A * N if kind == "masked" or c["lse"] else 0
    return {"bytes": 2 * 2.0 * A * N * D + 2 * 2.0 * S_tok * D + mask + lse,
            "flops": 4.0 * pairs * D}


def tolerance(c):
    kind = c["kind"]
    if kind == "gram":
        return {"rel": 1e-6}   # fp32 partial sums (4e-9 to 3e-8 off the 64-bit sums)
    if kind == "kv":
        return {"rel": 5e-3}   # one rounding to bf16 (1.4e-3 off)
    return {"rel": 1e-2}       # bf16 products, probabilities and outputs (2.2e-3 to 2.7e-3 off)


# ------------------------------------------------------------------------------ 64 bits
def _exact_attn(Q, K, V, frames, N, scale, O, lse=None, mask=None):
    """softmax(scale Q K^T) V of the given frames' rows in 64 bits into O [S_tok, H, d]."""
    S_tok, H, d = K.shape
    step = max(1, (1 << 26) // S_tok)
    rows = torch.cat([torch.arange(f * N, f * N + N, device=DEV) for f in frames])
    for h in range(H):
        q, k, v = Q[rows, h].double() * scale, K[:, h].double().t(), V[:, h].double()
        for r in range(0, len(rows), step):
            at = rows[r:r + step]
            s = q[r:r + step] @ k
            if mask is not None:
                ok = mask[h][at // 128].repeat_interleave(128, 1)[:, :S_tok]
                s.masked_fill_(ok == 0, -math.inf)
            m = s.amax(1, keepdim=True).clamp_min(-1e300)
            s = s.sub_(m).exp_()
            total = s.sum(1, keepdim=True)
            O[at, h] = (s @ v) / total.clamp_min(1e-300)
            if lse is not None:
                lse[h, at] = (m + total.log())[:, 0]


def _f64(*shape):
    return torch.zeros(*shape, dtype=torch.float64, device=DEV)


def _exact_step(c, row, z, v, Q, K, V, Kc, Vc, O, attn=True):
    """One step in place over 64-bit z, K, V and caches; returns the latent context."""
    F, N = c["F"], c["N"]
    ctx = torch.zeros_like(v, dtype=torch.float64)
    for f, (on, a, dt, slot) in enumerate(row):
        at = slice(f * N, f * N + N)
        ctx[f] = z[slot, f] if on else a * z[slot, f] + (1 - a) * z[1 - slot, f]
        for X, Xc in ((K, Kc), (V, Vc)):
            if on:
                Xc[1 - slot, f] = X[at].reshape(N, -1)
            else:
                X[at] = (a * Xc[slot, f] + (1 - a) * Xc[1 - slot, f]).view(N, c["H"], c["d"])
    if attn:
        _exact_attn(Q, K, V, [f for f, r in enumerate(row) if r[0]], N, 1.0 / math.sqrt(c["d"]),
                    O)
    for f, (on, a, dt, slot) in enumerate(row):
        if on:
            z[1 - slot, f] = z[slot, f] + dt * v[f].double()
    return ctx


def exact(c, seed):
    kind = c["kind"]
    t = _inputs(c, seed)
    if kind == "gram":
        F, E = t["P"].shape
        G = _f64(F, F)
        for e in range(0, E, 1 << 20):
            p = t["P"][:, e:e + (1 << 20)].double()
            G += p @ p.t()
        return {"G": G}
    F, N, H, d = c["F"], c["N"], c["H"], c["d"]
    if kind == "kv":
        out = {k: t[k].double() for k in ("K", "V", "Kc", "Vc")}
        on = _active_mask(F, c["A"])
        for f in range(F):
            a, slot = t["alpha"][f].double(), f % 2
            for k in ("K", "V"):
                X, Xc, at = out[k], out[k + "c"], slice(f * N, f * N + N)
                if on[f]:
                    Xc[1 - slot, f] = X[at].reshape(N, -1)
                else:
                    X[at] = (a * Xc[slot, f] + (1 - a) * Xc[1 - slot, f]).view(N, H, d)
        return out
    if work(c)["flops"] > EXACT_FLOPS and kind in ("attn", "masked", "step", "graph"):
        return None
    O = _f64(F * N, H, d)
    if kind == "masked" or kind == "attn":
        lse = _f64(H, F * N) if kind == "masked" or c["lse"] else None
        frames = [f for f, on in enumerate(_active_mask(F, c["A"])) if on]
        _exact_attn(t["Q"], t["K"], t["V"], frames, N, 1.0 / math.sqrt(d), O, lse,
                    t.get("mask"))
        return {"O": O, "lse": lse} if lse is not None else {"O": O}
    rows = _schedule(c)
    z, K, V = t["z"].double(), t["K"].double(), t["V"].double()
    Kc, Vc = t["Kc"].double(), t["Vc"].double()
    if kind == "step":
        ctx = _exact_step(c, rows[c["s"]], z, t["v"][0], t["Q"], K, V, Kc, Vc, O)
        return {"O": O, "ctx": ctx, "z": z, "K": K, "V": V, "Kc": Kc, "Vc": Vc}
    attn = work(c)["flops"] <= EXACT_FLOPS
    if kind == "graph":
        z[1] = z[0]
    Kc, Vc = Kc.repeat(2, 1, 1, 1), Vc.repeat(2, 1, 1, 1)
    for s, row in enumerate(rows):
        Q = t["Q"]
        if kind == "pipeline":  # each step's own host buffers
            Q, K, V = ((t["Q"], t["K"], t["V"]) if s % 2 == 0 else (t["Q2"], t["K2"], t["V2"]))
            K, V = K.double(), V.double()
        ctx = _exact_step(c, row, z, t["v"][s], Q, K, V, Kc, Vc, O, attn)
    if kind == "pipeline":
        return {"O": O if attn else None, "z": z, "ctx": ctx}
    return {"O": O, "ctx": ctx, "z": z, "K": K, "V": V, "Kc": Kc, "Vc": Vc}
