"""The calls whose time this repository is measured by.

Three calls make up a user's program: the draft step (``retrieve_fuse``, once
per draft-tree expansion of a decoding loop), the memory build
(``build_memory``, once per batch of images) and the LM head
(``lm_head_topk``, once per expansion).  The listed cases take each of them
through its public binding over the sizes of ``workloads.py`` and
``bench.py``: from the root and its six children against one image to
hundreds of draft states against 8192 entries each; full, padded and
scattered masks; flat, peaked and temperature-scaled rows; the paper's
retrieval settings; bf16 and fp32.  ``draw`` gives further cases of the same
ranges.

A step case: ``entries`` and ``rows`` hold one number per image (the valid
entries of its memory, the draft states that query it), ``pad`` the entries
of an image's visual tokens (valid ones first, or ``scatter``-ed), ``peaked``
the share of rows whose query points at one entry, ``hot`` whether every row
has a temperature in [0.1, 10], ``l_max`` the depth gate (-1: every row is
corrected), ``readout`` whether the caller asks for r.
"""

import math

import torch

from paper_2608_22883_gb300 import fovea

HIDDEN, DEPTH = 512, 6
LN_EPS, RMS_EPS = 1e-5, 1e-6


def _step(name, dtype, d, entries, rows, rho, k_min, k_max, **more):
    case = dict(name=name, kind="step", dtype=dtype, d=d, entries=entries, rows=rows, pad=0,
                scatter=False, rho=rho, k_min=k_min, k_max=k_max, peaked=0.0, hot=False,
                clusters=0, l_max=-1, readout=False)
    case.update(more)
    return case


def _build(name, dtype, d, entries, **more):
    case = dict(name=name, kind="build", dtype=dtype, d=d, entries=entries, pad=0, scatter=False,
                clusters=0)
    case.update(more)
    return case


def listed():
    return [
        # The first expansion of a tree: the root and its K_c = 6 children, one
        # image.  The smallest step of a decoding loop: latency and launches.
        _step("step-root-and-children", "bf16", 4096, "576", "7", 0.9, 1, 64, peaked=0.3),
        # One sequence's whole draft tree against one 576-token image.
        _step("step-one-image", "bf16", 4096, "576", "64", 0.9, 1, 64, peaked=0.125),
        # The paper's retrieval setting, with the depth gate of its setup open
        # to depth 2 and the readout returned (what a program that inspects the
        # evidence asks for).
        _step("step-paper-setting", "bf16", 4096, "576", "64", 0.8, 32, 256, peaked=0.125, l_max=2,
              readout=True),
        # Attention over the whole image: every entry selected.
        _step("step-dense", "bf16", 4096, "576", "64", 1.0, 576, 576),
        # A serving batch of variable-resolution images, padded to the longest,
        # a temperature per draft state.
        _step("step-ragged-batch", "bf16", 3584, "2880,1024,1024,1024,256,256,1024,2880",
              "32,32,32,32,32,32,32,32", 0.8, 1, 128, pad=2880, hot=True),
        # A full serving batch: 16 sequences of one wide model.
        _step("step-wide-batch", "bf16", 5120, ",".join(["576"] * 16), ",".join(["64"] * 16),
              0.95, 1, 64, peaked=0.125),
        # Long visual memories (video, many pages), clustered tokens.
        _step("step-long-memory", "bf16", 4096, "8192,8192,8192,8192", "128,128,128,128", 0.9, 1,
              256, clusters=64),
        # The fp32 path (checks against a full-precision pipeline; small models).
        _step("step-fp32", "fp32", 1024, "576,130", "33,31", 0.9, 1, 64, peaked=0.125),
        # Prefill of one image: the time to the first draft step.
        _build("build-one-image", "bf16", 4096, "576"),
        # Prefill of a serving batch of padded, partly masked images.
        _build("build-ragged-batch", "bf16", 3584, "2880,1024,1024,1024,256,256,1024,2880",
               pad=2880, scatter=True),
        # Prefill of long visual memories: the largest call.
        _build("build-long-memory", "bf16", 4096, "8192,8192,8192,8192", clusters=64),
        # Draft logits and the K_c = 6 tree candidates of one tree's states.
        dict(name="lm-head", kind="lm_head", vocab=32000, d=4096, rows=64, k_c=6, logits=True),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["step", "step", "step", "step", "build", "lm_head"])
    if kind == "lm_head":
        d = 64 * log_int(8, 80)
        rows = log_int(1, 128)
        vocab = log_int(2000, 32000 * 4096 // max(d, 4096))
        return dict(kind=kind, vocab=vocab, d=d, rows=rows, k_c=rng.choice([1, 4, 6, 6, 8, 10]),
                    logits=rng.random() < 0.6)
    fp32 = rng.random() < 0.15
    d = rng.choice([256, 512, 1024]) if fp32 else rng.choice([1024, 2048, 3584, 4096, 5120,
                                                              64 * log_int(8, 80)])
    images = rng.choice([1, 1, 1, 2, 3, 4, 8, 16])
    top = 700 if fp32 else min(8192, 32768 * 4096 ** 2 // (images * d * max(d, 4096)))
    entries = [log_int(24, top) for _ in range(images)]
    if rng.random() < 0.4:                       # one resolution for the whole batch
        entries = [entries[0]] * images
    pad = max(entries) + (rng.choice([0, 3, 40]) if rng.random() < 0.5 else 0)
    base = dict(dtype="fp32" if fp32 else "bf16", d=d, entries=",".join(map(str, entries)), pad=pad,
                scatter=rng.random() < 0.3, clusters=rng.choice([0, 0, 16, 64]))
    if kind == "build":
        return dict(kind="build", **base)
    most = 64 if fp32 else max(1, min(128, 1024 // images))
    rows = [log_int(1, most) for _ in range(images)]
    k_max = rng.choice([16, 64, 64, 128, 256, 256, log_int(300, 1024)])
    k_min = rng.choice([1, 1, min(32, k_max), k_max])
    return dict(kind="step", rows=",".join(map(str, rows)), rho=rng.choice([0.8, 0.9, 0.95]),
                k_min=k_min, k_max=k_max, peaked=rng.choice([0.0, 0.125, 0.5]),
                hot=rng.random() < 0.3, l_max=rng.choice([-1, -1, -1, 1, 2]),
                readout=rng.random() < 0.25, **base)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _numbers(text):
    return [int(x) for x in str(text).split(",")]


def _dtype(case):
    return torch.bfloat16 if case.get("dtype", "bf16") == "bf16" else torch.float32


def _weights(g, d, dt):
    def normal(*shape, scale=1.0, mean=0.0):
        return (torch.randn(shape, generator=g, device="cuda") * scale + mean).to(dt)

    H = HIDDEN
    return {
        "ln_v_gamma": normal(d, scale=0.1, mean=1.0), "ln_v_beta": normal(d, scale=0.1),
        "W_K": normal(d, d, scale=d ** -0.5), "W_U": normal(d, d, scale=d ** -0.5),
        "ln_h_gamma": normal(d, scale=0.1, mean=1.0), "ln_h_beta": normal(d, scale=0.1),
        "E_dep": normal(DEPTH + 1, d, scale=0.1), "W_Q": normal(d, d, scale=d ** -0.5),
        "W_f1": normal(H, 2 * d, scale=(2 * d) ** -0.5), "b_f1": normal(H, scale=0.01),
        "W_f2": normal(d, H, scale=H ** -0.5), "b_f2": normal(d, scale=0.01),
        "W_g1": normal(H, 2 * d, scale=(2 * d) ** -0.5), "b_g1": normal(H, scale=0.01),
        "w_g2": normal(H, scale=H ** -0.5), "b_g2": torch.zeros(1, device="cuda", dtype=dt),
        "rms_gamma": normal(d, scale=0.1, mean=1.0),
    }


def _images(case, g):
    """Visual tokens [B, M_max, d], the mask (None: every entry valid) and the
    valid positions of each image."""
    d, dt = case["d"], _dtype(case)
    entries = _numbers(case["entries"])
    B, M = len(entries), max(max(entries), case["pad"])
    if case["clusters"]:
        centres = torch.randn((case["clusters"], d), generator=g, device="cuda")
        z = torch.randint(0, case["clusters"], (B, M), generator=g, device="cuda")
        v = torch.empty((B, M, d), device="cuda", dtype=dt)
        for b in range(B):
            v[b] = (centres[z[b]] + 0.2 * torch.randn((M, d), generator=g, device="cuda")).to(dt)
    else:
        v = torch.empty((B, M, d), device="cuda", dtype=dt)
        for b in range(B):
            v[b] = torch.randn((M, d), generator=g, device="cuda").to(dt)
    if all(m == M for m in entries):
        return v, None, [torch.arange(M, device="cuda")] * B
    mask = torch.zeros((B, M), dtype=torch.uint8, device="cuda")
    valid = []
    for b, m in enumerate(entries):
        order = torch.randperm(M, generator=g, device="cuda") if case["scatter"] else torch.arange(M, device="cuda")
        valid.append(order[:m].sort().values)
        mask[b, valid[b]] = 1
    return v, mask, valid


def _layer_norm(x, gamma, beta):
    mean = x.mean(-1, keepdim=True)
    var = ((x - mean) ** 2).mean(-1, keepdim=True)
    return (x - mean) / torch.sqrt(var + LN_EPS) * gamma.to(x.dtype) + beta.to(x.dtype)


def _tree_depths(rows):
    return [0 if j == 0 else 1 if j <= 6 else 2 + (j - 7) % (DEPTH - 1) for j in range(rows)]


def _inputs(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    if case["kind"] == "lm_head":
        V, d = case["vocab"], case["d"]
        W = torch.empty((V, d), device="cuda", dtype=torch.bfloat16)
        for v0 in range(0, V, 8192):
            w = torch.randn((min(8192, V - v0), d), generator=g, device="cuda")
            W[v0:v0 + 8192] = (w * d ** -0.5).to(torch.bfloat16)
        h = torch.randn((case["rows"], d), generator=g, device="cuda").to(torch.bfloat16)
        return dict(W=W, h=h)
    d, dt = case["d"], _dtype(case)
    w = _weights(g, d, dt)
    v, mask, valid = _images(case, g)
    x = dict(w=w, v=v, mask=mask, valid=valid)
    if case["kind"] == "build":
        return x
    rows = _numbers(case["rows"])
    N = sum(rows)
    h = torch.randn((N, d), generator=g, device="cuda")
    r0 = 0
    for b, r in enumerate(rows):
        # peaked rows: part of h points along the query map's image of one key,
        # so that its score stands 5 to 20 above the rest
        n = min(r, int(round(r * case["peaked"])))
        if n:
            pick = valid[b][torch.randint(0, len(valid[b]), (n,), generator=g, device="cuda")]
            key = _layer_norm(v[b, pick].float(), w["ln_v_gamma"], w["ln_v_beta"]) @ w["W_K"].float().T
            along = key @ w["W_Q"].float()
            along = along / along.norm(dim=1, keepdim=True) * d ** 0.5
            a = 5.0 + 15.0 * torch.rand((n, 1), generator=g, device="cuda")
            h[r0:r0 + n] += a * d ** -0.5 * along
        r0 += r
    depth = torch.tensor([l for r in rows for l in _tree_depths(r)], dtype=torch.int32, device="cuda")
    scale = None
    if case["hot"]:
        t = torch.empty(N, device="cuda").uniform_(math.log(0.1), math.log(10.0), generator=g)
        scale = torch.exp(-t)
    offsets = [0]
    for r in rows:
        offsets.append(offsets[-1] + r)
    x.update(h=h.to(dt), depth=depth, row_scale=scale, offsets=offsets)
    return x


def prepare(case, seed):
    x = _inputs(case, seed)
    s = dict(case=case, **x)
    if case["kind"] == "lm_head":
        N = case["rows"]
        s["workspace"] = fovea.lm_head_workspace(case["vocab"], case["d"], N, case["k_c"])
        s["logits"] = (torch.empty((N, case["vocab"]), device="cuda") if case["logits"] else None)
        return s
    dtype = fovea.BF16 if case["dtype"] == "bf16" else fovea.FP32
    s["params"] = fovea.Params(x["w"], d_model=case["d"], mlp_hidden=HIDDEN, max_depth=DEPTH,
                               dtype=dtype, ln_eps=LN_EPS, rms_eps=RMS_EPS)
    if case["kind"] == "build":
        return s
    s["memory"] = fovea.build_memory(s["params"], x["v"], x["mask"])
    s["v"] = s["mask"] = None                    # a decoding loop keeps the memory alone
    N, d, k_max = x["offsets"][-1], case["d"], case["k_max"]
    s["workspace"] = fovea.new_workspace(s["params"], s["memory"], x["offsets"], k_max)
    s["out"] = dict(
        h_out=torch.empty_like(x["h"]),
        counts=torch.empty(N, dtype=torch.int32, device="cuda"),
        indices=torch.empty((N, k_max), dtype=torch.int32, device="cuda"),
        gate=torch.empty(N, device="cuda"),
        readout=torch.empty((N, d), device="cuda") if case["readout"] else None)
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "lm_head":
        idx, val, logits = fovea.lm_head_topk(s["W"], s["h"], case["k_c"], s["workspace"],
                                              logits=s["logits"], write_logits=case["logits"])
        return dict(index=idx, value=val, logits=logits)
    if case["kind"] == "build":
        memory = fovea.build_memory(s["params"], s["v"], s["mask"])
        keys, values, index, offsets = memory.views()
        out = dict(keys=keys, values=values, index=index, offsets=offsets,
                   folded=memory.folded_keys(s["params"]))
        for t in out.values():                   # the views live as long as the memory:
            if isinstance(t, torch.Tensor):      # each keeps it
                t.memory = memory
        return out
    out = s["out"]
    fovea.retrieve_fuse(s["params"], s["memory"], s["h"], s["depth"], s["offsets"], s["row_scale"],
                        case["rho"], case["k_min"], case["k_max"], out["h_out"], s["workspace"],
                        counts=out["counts"], indices=out["indices"], readout=out["readout"],
                        gate=out["gate"], l_max=None if case["l_max"] < 0 else case["l_max"])
    return out


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    """Each input read once, each output written once.  A step: the keys with
    W_Q, or the folded keys (two stored values per element), whichever is
    less; of the first fusion layer its h-half and 2H values per selected
    entry (at most every valid one); W_f2; the rows in and out.  A build: the
    valid tokens and the weights in, the stored tensors out."""
    d = case["d"]
    if case["kind"] == "lm_head":
        V, N, k = case["vocab"], case["rows"], case["k_c"]
        return {"bytes": 2.0 * V * d + 2.0 * N * d + (4.0 * N * V if case["logits"] else 0.0) + 8.0 * N * k,
                "flops": 2.0 * N * V * d}
    H = HIDDEN
    es = 2 if case["dtype"] == "bf16" else 4
    entries = _numbers(case["entries"])
    total = sum(entries)
    if case["kind"] == "build":
        folded = 2 * d if es == 2 else 0
        proj = 2 * H if es == 2 else 0
        return {"bytes": es * (total * d + 2.0 * d * d + (d * d + 2 * H * d if es == 2 else 0)
                               + total * (2.0 * d + folded + proj)) + 4.0 * total,
                "flops": 2.0 * total * d * (2 * d + (d + 2 * H if es == 2 else 0))}
    rows = _numbers(case["rows"])
    N = sum(rows)
    gated = case["l_max"] >= 0
    use = [sum(1 for l in _tree_depths(r) if not gated or l <= case["l_max"]) for r in rows]
    scored = sum(m for m, u in zip(entries, use) if u)
    picked = sum(min(m, u * case["k_max"]) for m, u in zip(entries, use))
    pairs = float(sum(m * u for m, u in zip(entries, use)))
    corrected = sum(use)
    if es == 2:
        fold = 2 * scored <= scored + d
        keys = 2.0 * scored * d if fold else (scored + d) * float(d)
        flops = 2.0 * pairs * d + (0.0 if fold else 2.0 * corrected * d * d)
        evidence, first = picked * 2.0 * H, 2.0 * H * d
    else:
        keys, flops = (scored + d) * float(d), 2.0 * pairs * d + 2.0 * corrected * d * d
        evidence, first = picked * float(d), 2.0 * H * 2 * d
    flops += 2.0 * corrected * (first + H * d)
    out = N * (4.0 + 4.0 * case["k_max"] + 4.0) + (4.0 * N * d if case["readout"] else 0.0)
    return {"bytes": es * (keys + evidence + first + d * H + 2.0 * N * d) + out, "flops": flops}


def tolerance(case):
    """About four times what two correct orders of the same sums showed: the
    steps scored through W_Q against the keys and against the folded keys; the
    LM head and the builds against 64 bits (a stored hi / lo pair splits
    differently where hi rounds the other way)."""
    if case["kind"] == "lm_head":
        return {"rel": 2e-5, "max": 1e-4, "differ": 0.004}
    if case["kind"] == "build":
        return {"rel": 3e-6, "max": 2e-5} if case["dtype"] == "fp32" else {"rel": 2e-3, "max": 0.2}
    if case["dtype"] == "fp32":
        return {"rel": 3e-6, "max": 2e-5, "differ": 0.004}
    return {"rel": 2e-3, "max": 0.06, "differ": 0.01}


# ---------------------------------------------------------------------------
# The same results in 64 bits
# ---------------------------------------------------------------------------

def _stored(x, dt):
    """x as the storage type holds it, in 64 bits."""
    return x.to(dt).double() if dt == torch.bfloat16 else x


def exact(case, seed):
    """Plain float64 in the paper's order, from the stored inputs.  In bf16
    the values that decide the selection (LN(v), k, u, LN(h) + E_dep) are
    rounded where the interface says they are stored; results are not."""
    x = _inputs(case, seed)
    if case["kind"] == "lm_head":
        z = x["h"].double() @ x["W"].double().T
        val, idx = torch.sort(z, dim=1, descending=True, stable=True)
        return dict(index=idx[:, :case["k_c"]].to(torch.int32), value=val[:, :case["k_c"]],
                    logits=z if case["logits"] else None)
    dt, d = _dtype(case), case["d"]
    w = x["w"]
    W = {n: t.double() for n, t in w.items()}
    keys, values = [], []
    for b, pos in enumerate(x["valid"]):
        lv = _stored(_layer_norm(x["v"][b, pos].double(), W["ln_v_gamma"], W["ln_v_beta"]), dt)
        keys.append(lv @ W["W_K"].T)
        values.append(lv @ W["W_U"].T)
    if case["kind"] == "build":
        offsets = [0]
        for k in keys:
            offsets.append(offsets[-1] + len(k))
        k = torch.cat(keys)
        folded = None
        if dt == torch.bfloat16:
            kappa = _stored(k, dt) @ W["W_Q"]
            hi = _stored(kappa, dt)
            folded = torch.cat([hi, kappa - hi], dim=1)
        return dict(keys=k, values=torch.cat(values), offsets=offsets, folded=folded,
                    index=torch.cat(x["valid"]).to(torch.int32))
    N, K_max = x["offsets"][-1], case["k_max"]
    h = x["h"].double()
    depth = x["depth"].long()
    q = _stored(_layer_norm(h, W["ln_h_gamma"], W["ln_h_beta"]) + W["E_dep"][depth], dt) @ W["W_Q"].T
    rho = float(torch.tensor(case["rho"], dtype=torch.float32))
    counts = torch.zeros(N, dtype=torch.int32, device="cuda")
    indices = torch.full((N, K_max), -1, dtype=torch.int32, device="cuda")
    r = torch.zeros((N, d), dtype=torch.float64, device="cuda")
    gated = (depth > case["l_max"]) if case["l_max"] >= 0 else torch.zeros_like(depth, dtype=torch.bool)
    for b, pos in enumerate(x["valid"]):
        lo, hi = x["offsets"][b], x["offsets"][b + 1]
        M = len(pos)
        if hi == lo or M == 0:
            continue
        s = q[lo:hi] @ _stored(keys[b], dt).T / math.sqrt(d)
        if x["row_scale"] is not None:
            s = s * x["row_scale"][lo:hi].double()[:, None]
        order_s, order = torch.sort(s, dim=1, descending=True, stable=True)
        mass = torch.cumsum(torch.softmax(order_s, dim=1), dim=1)
        k_raw = torch.where(mass[:, -1] >= rho, (mass < rho).sum(1) + 1, torch.full_like(depth[lo:hi], M))
        K = torch.clamp(k_raw, min=case["k_min"]).clamp(max=min(M, K_max))
        K = torch.where(gated[lo:hi], torch.zeros_like(K), K)
        m = min(M, K_max)
        take = torch.arange(m, device="cuda")[None, :] < K[:, None]
        a = torch.where(take, torch.exp(order_s[:, :m] - order_s[:, :1]), torch.zeros((), dtype=torch.float64, device="cuda"))
        a = a / a.sum(1, keepdim=True).clamp(min=1e-300)
        dense = torch.zeros_like(s).scatter_(1, order[:, :m], a)
        r[lo:hi] = dense @ _stored(values[b], dt)
        counts[lo:hi] = K.to(torch.int32)
        ids = pos[order[:, :m]].to(torch.int32)
        indices[lo:hi, :m] = torch.where(take, ids, torch.full_like(ids, -1))
    hr = torch.cat([h, r], dim=1)
    a_f = torch.nn.functional.silu(hr @ W["W_f1"].T + W["b_f1"])
    a_g = torch.nn.functional.silu(hr @ W["W_g1"].T + W["b_g1"])
    c = a_f @ W["W_f2"].T + W["b_f2"]
    gate = torch.sigmoid(a_g @ W["w_g2"] + W["b_g2"])
    y = h + gate[:, None] * c
    out = y / torch.sqrt((y * y).mean(1, keepdim=True) + RMS_EPS) * W["rms_gamma"]
    return dict(h_out=torch.where(gated[:, None], h, out), counts=counts, indices=indices,
                gate=torch.where(gated, torch.zeros_like(gate), gate),
                readout=r if case["readout"] else None)
