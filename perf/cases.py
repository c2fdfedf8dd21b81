"""The work that users of this library have it do, as measurable cases.

A case is a dict of plain values; prepare() builds from it what a serving program has in hand before the call
(tensors on the GPU, a context with its workspace, a recorded graph), run() is one pass through the public entry
points of paper_2504_08966_b200.binding, and its outputs come back whole.

Keys of a case
    call     which entry points: "reduce" (pact_reduce), "graph" (pact_graph_launch of a recorded pact_reduce),
             "host" (pact_reduce_host on pinned host buffers), "stages" (the five stage calls one after the other),
             "euti" (pact_importance + pact_prune), "cluster" (pact_dbdpc over all tokens + pact_merge),
             "spread" (pact_key_spread over `layers` key matrices)
    B, N, T  images in the call, visual tokens of the largest one, text tokens of each; `ragged`: the images of the
             call have different sizes and parameters of their own
    d, n_qh, n_kvh, d_h   hidden size, query heads, key heads, head width
    dtype, out            element types of the inputs and of the merged rows ("bf16" or "fp32")
    scene    what the images look like, see _latents()
    blobs    distinct image regions of an image
    lam, d_c pruning fraction and clustering cutoff
    rope     the clustering keys are a second buffer (after the rotary embedding), not the scoring keys themselves

The inputs follow the recipes of paper_2504_08966_b200/workloads.py, drawn on the GPU.
"""
import math

import torch

from paper_2504_08966_b200 import binding as pb

_TYPES = {"bf16": torch.bfloat16, "fp32": torch.float32}
_COUNTS = ("n_out", "q", "C", "r", "discarded")      # the first five counters, see prepare()

_BASE = {"call": "reduce", "B": 1, "N": 7290, "T": 64, "ragged": False, "d": 3584, "n_qh": 4, "n_kvh": 4, "d_h": 128,
         "dtype": "bf16", "out": "bf16", "scene": "photo", "blobs": 200, "lam": 0.5, "d_c": 0.3, "rope": False,
         "layers": 1}


def _case(name=None, **kw):
    c = dict(_BASE, **kw)
    return c if name is None else dict(c, name=name)


def listed():
    return [
        # the smallest call: a thumbnail on a small fp32 model; latency and launches are all there is
        _case("thumbnail_fp32", N=196, T=16, d=896, n_qh=2, n_kvh=2, d_h=64, dtype="fp32", out="fp32", scene="blobs",
              blobs=12, lam=0.3, d_c=0.4),
        # one crop (27 x 27 patches) of a chat request, a new pact_reduce call for every request
        _case("crop_729", N=729, T=32, blobs=60),
        # the benchmark's image (10 crops x 729): a server that keeps its buffers and replays the recorded step
        _case("image_7290_graph", call="graph"),
        # the same image given as host buffers, copies included (what an application without resident tensors pays)
        _case("image_7290_host", call="host"),
        # 32 frames x 196 tokens of a video, called directly
        _case("video_6272", N=6272, scene="video", blobs=40),
        # a batch of 16 requests of 4 crops each
        _case("batch_16x2916", B=16, N=2916, T=32, blobs=225),
        # three requests of different sizes and settings on a grouped-query model, with keys before and after the
        # rotary embedding and merged rows in fp32 for a consumer that goes on in fp32
        _case("ragged_gqa_3x2309", B=3, N=2309, T=40, ragged=True, n_qh=28, out="fp32", blobs=60, rope=True),
        # the largest call: four very long sequences with heavy-tailed norms and exact duplicates
        _case("long_4x16384", B=4, N=16384, scene="blobs", blobs=1000, lam=0.7, d_c=0.25),
        # the five steps one by one, for a program that looks at the intermediate results
        _case("stages_2500", call="stages", N=2500, T=20, blobs=70),
        # scoring and pruning alone (EUTI as a pruning method of its own)
        _case("euti_7290", call="euti"),
        # clustering and merging alone, nothing pruned (DBDPC as a clustering method of its own)
        _case("cluster_7290", call="cluster", lam=0.0),
        # the choice of the reduction layer from the keys of ten layers
        _case("layers_10x7290", call="spread", layers=10),
    ]


# (d, n_qh, n_kvh, d_h) of the models a caller may bring
_MODELS = [(896, 2, 2, 64), (896, 14, 2, 64), (2048, 16, 4, 128), (3584, 4, 4, 128), (3584, 28, 4, 128),
           (3072, 32, 8, 96), (4096, 32, 8, 128)]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges."""
    call = rng.choices(["reduce", "graph", "host", "stages", "euti", "cluster", "spread"],
                       [40, 15, 10, 10, 10, 7, 8])[0]
    d, n_qh, n_kvh, d_h = rng.choices(_MODELS, [1, 1, 1, 4, 2, 1, 1])[0]
    kw = {"call": call, "d": d, "n_qh": n_qh, "n_kvh": n_kvh, "d_h": d_h, "T": rng.randint(0, 96),
          "scene": rng.choices(["photo", "video", "blobs"], [3, 1, 1])[0],
          "lam": rng.choice([0.3, 0.5, 0.55, 0.7]), "d_c": rng.choice([0.2, 0.21, 0.25, 0.3, 0.5])}
    d_k, cols = n_kvh * d_h, n_qh * d_h
    if call in ("reduce", "graph"):
        if rng.random() < 0.15:                       # fp32 inputs: small models and images
            kw.update(dtype="fp32", d=896, n_qh=2, n_kvh=2, d_h=64, N=_log_int(rng, 32, 2500))
        else:
            B = kw["B"] = rng.choices([1, _log_int(rng, 2, 16)], [3, 2])[0]
            # no more bytes and no more distances than the largest listed case
            tokens = 65536 * 4608 // (d + d_k + cols)
            pairs = 9832 * math.sqrt(512 / (B * d_k)) / (1 - kw["lam"])
            kw["N"] = _log_int(rng, 48, int(min(16384, tokens // B, pairs)))
            kw["ragged"] = B > 1 and rng.random() < 0.5
        kw["out"] = "fp32" if kw.get("dtype") == "fp32" or rng.random() < 0.2 else "bf16"
        kw["rope"] = rng.random() < 0.4
    elif call == "spread":
        kw["layers"] = _log_int(rng, 1, 10)
        kw["N"] = _log_int(rng, 64, int(7290 * min(1.0, math.sqrt(512 / d_k))))
    elif call == "cluster":
        kw["N"] = _log_int(rng, 64, int(7290 * min(1.0, math.sqrt(512 / d_k))))
        kw["lam"] = 0.0
    else:
        kw["N"] = _log_int(rng, 64, min(7290, 7290 * 4608 // (d + d_k + cols)))
    kw["blobs"] = max(2, min(1000, int(kw["N"] * rng.uniform(0.02, 0.08))))
    return _case(**kw)


# ---- inputs ------------------------------------------------------------------------------------------------------

def _sizes(case):
    """Visual tokens of each image of the call."""
    B, N = case["B"], case["N"]
    if not case["ragged"]:
        return [N] * B
    return [max(1, N - (N * b * 3) // (4 * B) - b) for b in range(B)]


def _settings(case, b):
    """(lam, d_c, alpha) of image b: per-image settings where the images differ."""
    if not case["ragged"]:
        return case["lam"], case["d_c"], 1.5
    return min(0.9, case["lam"] + 0.1 * (b % 3)), case["d_c"] + 0.05 * (b % 2), (1.5, 1.0, 2.0)[b % 3]


def _unit(x):
    return x / x.norm(dim=1, keepdim=True)


def _latents(g, scene, n, d_k, blobs):
    """n latent vectors and hidden-state norms.
    photo   half of the tokens in `blobs` image regions, 30 % near-duplicates, 20 % low-norm background
    video   frames of up to 196 tokens, each the one before plus noise, a tenth of the positions new
    blobs   regions of different spread, heavy-tailed norms, 1 % exact duplicates"""
    dev = {"device": "cuda", "generator": g}
    centres = _unit(torch.randn(blobs, d_k, **dev))
    s = 1.0 / math.sqrt(d_k)
    norms = torch.exp(0.5 * torch.randn(n, **dev))

    def blob(m, sig):
        which = torch.randint(blobs, (m,), **dev)
        return centres[which] + torch.randn(m, d_k, **dev) * (sig[which, None] * s)

    if scene == "video":
        per = min(n, 196)
        sig = torch.full((blobs,), 0.15, device="cuda")
        cur, frames = blob(per, sig), []
        for _ in range(-(-n // per)):
            frames.append(cur)
            moved = torch.rand(per, 1, **dev) < 0.1
            cur = torch.where(moved, blob(per, sig), cur + torch.randn(per, d_k, **dev) * (0.05 * s))
        return torch.cat(frames)[:n], norms, None
    if scene == "blobs":
        z = blob(n, 0.05 + 0.45 * torch.rand(blobs, **dev) if blobs > 100 else torch.full((blobs,), 0.15, device="cuda"))
        if blobs > 100:                               # Student-t with three degrees of freedom
            chi = torch.randn(n, 3, **dev).square().sum(1)
            norms = torch.randn(n, **dev).abs() / torch.sqrt(chi / 3) + 0.01
        dst = torch.randperm(n, **dev)[: n // 100]
        src = torch.randint(n, (n // 100,), **dev)
        return z, norms, (dst, src)
    n_blob, n_dup = n // 2, (3 * n) // 10
    sig = 0.1 + 0.2 * torch.rand(blobs, **dev)
    back = _unit(torch.randn(1, d_k, **dev)) + torch.randn(n - n_blob - n_dup, d_k, **dev) * s
    base = torch.cat([blob(n_blob, sig), back])
    low = torch.cat([torch.zeros(n_blob, device="cuda"), torch.ones(back.shape[0], device="cuda")])
    src = torch.randint(base.shape[0], (n_dup,), **dev)
    z = torch.cat([base, base[src] + torch.randn(n_dup, d_k, **dev) * (0.02 * s)])
    low = torch.cat([low, torch.zeros(n_dup, device="cuda")])
    perm = torch.randperm(n, **dev)
    z, low = z[perm], low[perm]
    return z, torch.where(low > 0, 0.05 * norms, norms), None


def _tensors(g, case, n):
    """H, K, Q, K_clu, P of one image."""
    d, d_k, cols, T = case["d"], case["n_kvh"] * case["d_h"], case["n_qh"] * case["d_h"], case["T"]
    dev = {"device": "cuda", "generator": g}
    dt = _TYPES[case["dtype"]]
    z, norms, dup = _latents(g, case["scene"], n, d_k, min(case["blobs"], n))
    R_q, R_h = torch.randn(d_k, cols, **dev) / math.sqrt(d_k), torch.randn(d_k, d, **dev) / math.sqrt(d_k)
    K = (z * torch.exp(0.25 * torch.randn(n, 1, **dev))).to(dt)
    Q = (z @ R_q + 0.1 * torch.randn(n, cols, **dev)).to(dt)
    H = torch.empty(n + T, d, dtype=dt, device="cuda")
    t0 = T // 4
    H[:t0] = torch.randn(t0, d, **dev)
    H[t0 + n:] = torch.randn(T - t0, d, **dev)
    H[t0:t0 + n] = _unit(z @ R_h) * norms[:, None]
    if dup is not None:
        dst, src = dup
        K[dst], Q[dst], H[t0 + dst] = K[src], Q[src], H[t0 + src]
    Kc = K
    if case["rope"]:                                  # a fixed rotation of the keys stands in for the embedding
        v = _unit(torch.randn(1, d_k, **dev))
        Kc = (K.float() - 2.0 * (K.float() @ v.T) @ v).to(dt)
    return H, K, Q, Kc, torch.arange(n + T, dtype=torch.int32, device="cuda"), t0


def _device_image(g, case, n):
    H, K, Q, Kc, P, t0 = _tensors(g, case, n)
    nt, out = n + case["T"], _TYPES[case["out"]]
    z = lambda m, dt: torch.zeros(m, dtype=dt, device="cuda")   # noqa: E731  rows past the last one stay zero
    return pb.DeviceImage(H, K, Q, Kc, P, t0, n, z((nt, case["d"]), out), z(nt, torch.int32), z(nt, torch.int32),
                          z(n, torch.int32), z(n, torch.float32), z(n, torch.uint8), z(pb.N_COUNTERS, torch.int32),
                          z(nt, torch.float32))


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    call, N = case["call"], case["N"]
    ctx = pb.Context(case["d"], case["n_qh"], case["n_kvh"], case["d_h"], _TYPES[case["dtype"]], _TYPES[case["out"]])
    st = {"call": call, "ctx": ctx}
    if call == "spread":
        d_k = case["n_kvh"] * case["d_h"]
        st["K"] = []
        for layer in range(case["layers"]):          # keys spread wider with depth, not monotonically
            mix = (0.02, 0.05, 0.04, 0.15, 0.4, 0.3, 0.9, 0.7, 1.5, 1.2)[layer % 10]
            k = _unit(torch.randn(1, d_k, device="cuda", generator=g)) + torch.randn(N, d_k, device="cuda", generator=g) * (mix / math.sqrt(d_k))
            st["K"].append((k * torch.exp(0.25 * torch.randn(N, 1, device="cuda", generator=g))).to(_TYPES[case["dtype"]]))
        st["out"] = [torch.zeros(case["layers"], dtype=torch.float32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")]
        ctx.ensure_workspace(min(case["layers"], 16), N)
        return st
    sizes = _sizes(case)
    params = []
    for b in range(case["B"]):
        lam, d_c, alpha = _settings(case, b)
        params.append(pb.make_params(lam=lam, d_c=d_c, alpha=alpha))
    st["params"] = params if case["ragged"] else params[0]
    if call == "host":
        H, K, Q, Kc, P, t0 = (x.cpu().pin_memory() if torch.is_tensor(x) else x for x in _tensors(g, case, N))
        nt = N + case["T"]
        z = lambda m, dt: torch.zeros(m, dtype=dt).pin_memory()   # noqa: E731
        h = dict(H=H, K_euti=K, Q_euti=Q, K_clu=Kc if case["rope"] else K, P=P, vis_start=t0, N=N, H_out=z((nt, case["d"]), _TYPES[case["out"]]),
                 P_out=z(nt, torch.int32), size_out=z(nt, torch.int32), logw_out=z(nt, torch.float32), label=z(N, torch.int32),
                 counters=z(pb.N_COUNTERS, torch.int32))
        st["host"] = h
        st["staging"] = torch.empty(ctx.host_staging_bytes(nt, N), dtype=torch.uint8, device="cuda")
        ctx.ensure_workspace(1, N)
        st["out"] = [h["H_out"], h["P_out"], h["size_out"], h["logw_out"], h["label"], h["counters"][:len(_COUNTS)]]
        return st
    st["images"] = ims = [_device_image(g, case, n) for n in sizes]
    ctx.ensure_workspace(case["B"], max(sizes))
    if call == "graph":
        st["graph"] = ctx.pact_graph_create(ims, st["params"])
    # The counters come back as far as they are results: the number of sweeps behind them depends on timing.
    # With more images than a reader wants tensors for, the merged rows of all come back and the rest of the first.
    st["out"] = [[im.H_out, im.label, im.size_out] for im in ims] + [
        [im.P_out, im.logw_out, im.score, im.keep, im.counters[:len(_COUNTS)]] for im in ims[:2]]
    if call in ("stages", "euti", "cluster"):
        i32 = lambda n: torch.zeros(n, dtype=torch.int32, device="cuda")   # noqa: E731
        im = ims[0]
        st.update(kept=i32(N), pruned=i32(N), counts=i32(2), rho=torch.zeros(N, dtype=torch.float32, device="cuda"), centers=i32(N), C=i32(1), r=i32(1))
        st["q"], st["m"] = st["counts"][:1], st["counts"][1:]
        euti = [im.score, im.keep, st["kept"], st["pruned"], st["counts"]]
        rest = [st["rho"], st["centers"], st["C"], im.label, im.H_out, im.P_out, im.size_out, im.logw_out]
        if call == "euti":
            st["out"] = euti
        elif call == "stages":
            st["out"] = euti + [st["r"]] + rest
        else:
            st["kept"], st["q"] = torch.arange(N, dtype=torch.int32, device="cuda"), torch.full((1,), N, dtype=torch.int32, device="cuda")
            st["out"] = rest
    return st


# ---- one pass ----------------------------------------------------------------------------------------------------

def run(st):
    ctx, call = st["ctx"], st["call"]
    if call == "reduce":
        ctx.pact_reduce(st["images"], st["params"])
    elif call == "graph":
        st["graph"].launch()
    elif call == "host":
        ctx.pact_reduce_host(st["host"], st["params"], st["staging"])
    elif call == "spread":
        ctx.pact_key_spread(st["K"], 0.3, st["out"][0], st["out"][1])
    else:
        im, p = st["images"][0], st["params"]
        if call != "cluster":
            ctx.pact_importance(im, p, im.score)
            ctx.pact_prune(im.score, p, im.keep, st["kept"], st["pruned"], st["counts"])
        if call != "euti":
            ctx.pact_dbdpc(im.K_clu, st["kept"], st["q"], p, st["rho"], st["centers"], st["C"], im.label)
            if call == "stages":
                ctx.pact_reincorporate(im.K_clu, st["pruned"], st["m"], st["centers"], st["C"], p, im.label, st["r"])
            ctx.pact_merge(im, im.label, st["centers"], st["C"], p)
    return st["out"]


# ---- what a pass cannot do without -------------------------------------------------------------------------------

def work(case):
    call, e, oe = case["call"], 2 if case["dtype"] == "bf16" else 4, 2 if case["out"] == "bf16" else 4
    d, d_k, cols, T = case["d"], case["n_kvh"] * case["d_h"], case["n_qh"] * case["d_h"], case["T"]
    if call == "spread":
        L, N = case["layers"], case["N"]
        return {"bytes": L * (N * d_k * e + 4.0), "flops": L * float(d_k) * N * (N - 1)}
    bytes_ = flops = 0.0
    for b, N in enumerate(_sizes(case)):
        q = N - int(_settings(case, b)[0] * N)
        # clusters: about the image regions, and on photos a part of the scattered background
        C = min(q, min(case["blobs"], N) + (N // 25 if case["scene"] == "photo" else 0))
        if call != "cluster":                         # scores and split: H, K and Q in, score, keep flag and list entry out
            bytes_ += N * (d + d_k + cols) * e + 9.0 * N
            flops += 2.0 * N * (d + d_k * (case["n_qh"] // case["n_kvh"]) + cols)
        if call == "euti":
            continue
        if call == "cluster" or case["rope"]:
            bytes_ += N * d_k * e                     # the clustering keys, where scoring has not read them
        if call == "cluster":
            bytes_ += N * d * e
        # labels, ids in, merged rows, ids, sizes and their logarithms out, text rows copied
        bytes_ += 4.0 * N + 4.0 * (N + T) + C * (d * oe + 12.0) + T * (d * (e + oe) + 12.0)
        flops += float(d_k) * q * (q + 1) + 2.0 * d_k * N * C + N * d
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    # Keep flags, labels, lists, ids and sizes are whole numbers of a uniquely defined result.  Merged rows: bf16 holds
    # eight bits, fp32 sums are good to about 1e-5.  Key distances come from fp32 sums of d_k products.
    if case["call"] == "spread":
        return {"rel": 3e-5, "max": 2e-4}
    if case["call"] == "euti":
        return {"rel": 1e-5}
    return {"rel": 4e-3, "max": 2e-2} if case["out"] == "bf16" else {"rel": 1e-5, "max": 4e-4}
