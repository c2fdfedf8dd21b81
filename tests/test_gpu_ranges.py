"""Sizes at which a kernel's split of the work has its edges: ranges of the merge, units of the token pass, images of
the one-cluster step and of the kernels that take over from it."""
import numpy as np
import pytest
import torch

from paper_2504_08966_b200 import workloads
from tests.helpers import compare_image, fragile_report, gpu_reduce, oracle_image

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,C,T,d,dtype", [
    (1, 1, 0, 3584, torch.bfloat16), (17, 1, 0, 3584, torch.bfloat16), (31, 31, 2, 520, torch.bfloat16),
    (300, 1, 5, 896, torch.float32),          # one cluster over all ranges
    (1184, 9, 3, 1032, torch.float32),        # a last slice of one vector
    (2909, 37, 64, 3584, torch.bfloat16), (4737, 2, 0, 8192, torch.bfloat16),
    (7301, 700, 64, 8, torch.bfloat16),
    (20011, 41, 7, 3584, torch.bfloat16),     # two vectors per thread
])
def test_merge_ranges(N, C, T, d, dtype):
    """Clusters that end inside a range of members, cross one boundary, or cover many; some tokens in no cluster."""
    from paper_2504_08966_b200 import binding as pb
    g = torch.Generator(device="cuda").manual_seed(N)
    H = torch.randn(N + T, d, device="cuda", generator=g).to(dtype)
    label = torch.randint(-1 if N > 40 else 0, C, (N,), device="cuda", generator=g, dtype=torch.int32)
    label[label == C // 2] = 0                # one large cluster, one without members but its centre
    cidx = torch.arange(C, dtype=torch.int32, device="cuda")
    label[:C] = cidx
    n = N + T
    z = lambda m, dt: torch.zeros(m, dtype=dt, device="cuda")   # noqa: E731
    K = z((N, 64), dtype)
    im = pb.DeviceImage(H, K, K, K, torch.arange(n, dtype=torch.int32, device="cuda"), T // 2, N, z((n, d), torch.float32), z(n, torch.int32),
                        z(n, torch.int32), z(N, torch.int32), z(N, torch.float32), z(N, torch.uint8), z(pb.N_COUNTERS, torch.int32), z(n, torch.float32))
    ctx = pb.Context(d, 1, 1, 64, dtype, torch.float32)
    for _ in range(2):                        # the tickets of the first call must not be left over
        ctx.pact_merge(im, label, cidx, torch.tensor([C], dtype=torch.int32, device="cuda"), pb.make_params())
    torch.cuda.synchronize()
    v0, lab = T // 2, label.long()
    keep = lab >= 0
    size = torch.bincount(lab[keep], minlength=C)
    want = torch.zeros(C, d, dtype=torch.float64, device="cuda").index_add_(0, lab[keep], H[v0:v0 + N][keep].double()) / size[:, None]
    assert int(im.counters[0]) == C + T and int(im.counters[pb.CNT["status"]]) == 0
    assert torch.equal(im.size_out[v0:v0 + C].long(), size)
    err = (im.H_out[v0:v0 + C].double() - want).abs().amax(1) / want.abs().amax(1)
    assert float(err.max()) < 2e-5
    text = torch.cat([im.H_out[:v0], im.H_out[v0 + C:C + T]])
    assert torch.equal(text, torch.cat([H[:v0], H[v0 + N:]]).float())


def _workload(N, n_qh, n_kvh, d_h, d, dtype, seed, scale=1.0, rope=False, T=3):
    rng = np.random.default_rng(seed)
    dk = n_kvh * d_h
    t = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(torch.float32).to(dtype)   # noqa: E731
    blobs = rng.standard_normal((max(1, N // 12), dk))
    z = blobs[rng.integers(0, blobs.shape[0], N)] + 0.25 * rng.standard_normal((N, dk))
    R = rng.standard_normal((dk, n_qh * d_h)) / np.sqrt(dk)
    K = t(scale * z)
    img = workloads.Image(H=t(rng.standard_normal((N + T, d)) * np.exp(0.5 * rng.standard_normal((N + T, 1)))), K=K, Q=t(z @ R), P=torch.arange(N + T, dtype=torch.int32),
                          n_total=N + T, vis_start=1, N=N, K_clu=t(z + 0.05 * rng.standard_normal((N, dk))) if rope else None)
    return workloads.Workload("edge", [img], d, n_qh, n_kvh, d_h, dtype, 0.5, 0.3)


def _check(wl, out_dtype):
    outs, _ = gpu_reduce(wl, out_dtype)
    for img, g in zip(wl.images, outs):
        o = oracle_image(wl, img)
        bad = compare_image(o, g, img, out_dtype == torch.bfloat16)
        assert not bad, f"{bad}; fragile: {fragile_report(o, wl.d_c, wl.alpha)}"


@pytest.mark.parametrize("N,n_qh,n_kvh,d_h,d,dtype,scale,rope", [
    (1, 1, 1, 8, 8, torch.bfloat16, 1.0, False), (7, 2, 2, 64, 896, torch.float32, 1.0, False),
    (9, 3, 1, 40, 72, torch.bfloat16, 1.0, True),                 # three heads of one key head, five vectors per head
    (1185, 5, 1, 96, 136, torch.bfloat16, 1.0, False),            # units of nine tokens; heads in blocks of four and one
    (2369, 14, 2, 64, 896, torch.bfloat16, 4.0, False),           # seventeen tokens; four and three heads; steep softmax
    (4737, 28, 4, 128, 512, torch.bfloat16, 1.0, True),
    (1500, 4, 4, 36, 4104, torch.float32, 1.0, False),            # rows in three copies
    (4800, 2, 2, 12, 264, torch.float32, 1.0, True),
    (1200, 40, 40, 64, 1024, torch.bfloat16, 1.0, False),         # more heads than one block of the scoring kernel
])
def test_token_units(N, n_qh, n_kvh, d_h, d, dtype, scale, rope):
    _check(_workload(N, n_qh, n_kvh, d_h, d, dtype, N, scale, rope), torch.float32)


@pytest.mark.parametrize("N,n_qh,n_kvh,d_h,d,dtype", [
    (43, 64, 8, 128, 8192, torch.bfloat16), (2369, 64, 8, 128, 8192, torch.bfloat16),    # rows in halves beside the keys: units of eight and nine
    (301, 32, 8, 128, 4096, torch.float32), (1185, 16, 16, 128, 8192, torch.bfloat16),
    (301, 128, 8, 128, 8192, torch.bfloat16), (9, 96, 32, 96, 8192, torch.float32),       # no room for the keys: grouped heads, eight tokens
    (301, 40, 40, 128, 8192, torch.bfloat16),                                            # ... one head per key head
])
def test_wide_keys_and_queries(N, n_qh, n_kvh, d_h, d, dtype):
    """Models whose keys, global query and hidden states do not fit an SM's shared memory together."""
    _check(_workload(N, n_qh, n_kvh, d_h, d, dtype, N + d), torch.float32)


@pytest.mark.parametrize("N,n_qh,n_kvh,d_h,dtype", [
    (2368, 8, 1, 64, torch.bfloat16), (2369, 3, 1, 64, torch.bfloat16),       # units of eight and nine tokens: one block of eight, two
    (4736, 18, 2, 40, torch.bfloat16), (4737, 6, 2, 64, torch.float32),       # sixteen, seventeen; nine heads: eight and one
    (7104, 8, 2, 16, torch.float32), (7105, 28, 4, 32, torch.bfloat16),       # twenty-four, twenty-five
    (1700, 9, 3, 20, torch.float32),                                          # heads of five fours: the last step has half of its elements
    (777, 256, 2, 8, torch.bfloat16), (2600, 33, 11, 8, torch.bfloat16),      # more heads per CTA of the merge than warps, more than 32 in all
])
def test_heads_of_a_key_head_together(N, n_qh, n_kvh, d_h, dtype):
    """Three and more query heads per key head go through the double-precision tensor instruction, eight tokens at a time."""
    _check(_workload(N, n_qh, n_kvh, d_h, 64, dtype, 3 * N + 1), torch.float32)


@pytest.mark.parametrize("dtype,n_qh,n_kvh,d_h", [(torch.bfloat16, 4, 2, 64), (torch.bfloat16, 3, 3, 24), (torch.float32, 2, 2, 20)])
@pytest.mark.parametrize("N", [1, 2, 15, 17, 127, 129, 511, 513, 1023, 1024, 1025])
def test_small_images(N, dtype, n_qh, n_kvh, d_h):
    """Around the tiles and the limits of the one-cluster step; widths that the tensor cores take and others."""
    _check(_workload(N, n_qh, n_kvh, d_h, 256, dtype, 7 * N + 1), torch.float32)


@pytest.mark.parametrize("B", [2, 9, 16])
def test_small_batches(B):
    """As many images as clusters fit on the GPU at once, and more."""
    wls = [_workload(max(1, 300 - 19 * b), 4, 2, 64, 256, torch.bfloat16, 900 + b) for b in range(B)]
    wl = workloads.Workload("edge", [w.images[0] for w in wls], 256, 4, 2, 64, torch.bfloat16, 0.5, 0.3)
    _check(wl, torch.bfloat16)


def test_pairs_of_ctas_with_ragged_ends():
    """The all-pairs pass on pairs of CTAs (sixteen images of eleven blocks): last columns at every place in a word and a pair of words."""
    wls = [_workload(1281 + 13 * b, 2, 1, 64, 64, torch.bfloat16, 60 + b) for b in range(16)]
    wl = workloads.Workload("edge", [w.images[0] for w in wls], 64, 2, 1, 64, torch.bfloat16, 0.0, 0.3)
    _check(wl, torch.float32)


@pytest.mark.parametrize("N", [3072, 3073, 8192, 8193])
def test_select_key_registers(N):
    """The last sizes with the keys of the split in six and in sixteen registers per thread, and the ones after them."""
    _check(_workload(N, 2, 1, 16, 32, torch.bfloat16, N), torch.float32)


@pytest.mark.parametrize("N,d_h", [(1500, 64), (3100, 512), (9000, 64), (16384, 64), (16385, 64), (24577, 64)])
@pytest.mark.parametrize("same", [1, 2, 40, 300, 10 ** 6])
def test_split_with_equal_scores(N, d_h, same):
    """`same` tokens with each score: one key, a few or many under the threshold's prefix, and all; a tenth are zero, then most."""
    from paper_2504_08966_b200 import binding as pb
    g = torch.Generator().manual_seed(N + same)
    ctx = pb.Context(64, 1, 1, d_h, torch.bfloat16, torch.float32)
    for zeros, lam in ((0.1, 0.95), (0.1, 0.05), (0.7, 0.8)):
        # norms: one element per row, of more values than bf16 has between two powers of two
        a = torch.exp(1.5 * torch.randn(N // same + 1, generator=g))[torch.arange(N) // same % (N // same + 1)][torch.randperm(N, generator=g)]
        a[torch.rand(N, generator=g) < zeros] = 0.0
        H = torch.zeros(N, 64)
        for k in range(3):                        # a row's norm in three pieces of eight bits
            H[:, k] = (a - H[:, :k].sum(1)).to(torch.bfloat16).float()
        img = workloads.Image(H=H.to(torch.bfloat16), K=torch.randn(N, d_h, generator=g).to(torch.bfloat16), Q=torch.zeros(N, d_h, dtype=torch.bfloat16),
                              P=torch.arange(N, dtype=torch.int32), n_total=N, vis_start=0, N=N)
        im = pb.device_image(img, torch.float32)
        ctx.pact_reduce([im], pb.make_params(lam=lam, d_c=1.9, flags=pb.FLAG_NORM_ONLY))
        torch.cuda.synchronize()
        score = im.score.cpu().numpy()
        want = np.linalg.norm(H.numpy().astype(np.float64), axis=1) / N
        assert (np.abs(score - want) <= 2e-7 * want).all()
        keep = score >= np.sort(score)[int(np.floor(lam * N + 1e-6))]
        assert np.array_equal(im.keep.cpu().numpy(), keep)
        assert int(im.counters[pb.CNT["q"]]) == keep.sum() and int(im.counters[pb.CNT["status"]]) == 0


@pytest.mark.parametrize("N", [1, 2, 31, 33, 511, 513, 3072, 3073, 8192, 8193, 16384, 16385])
@pytest.mark.parametrize("kind", ["spread", "signs", "tenths", "pairs", "hundreds", "one value", "infinities"])
def test_split_of_given_scores(N, kind):
    """pact_prune around the sizes of its kernels: one, a few and many candidates under a prefix, keys that differ in every bit."""
    from oracle import pact_oracle as orc
    from paper_2504_08966_b200 import binding as pb
    rng = np.random.default_rng(N)
    x = {"spread": lambda: np.exp(3 * rng.standard_normal(N)), "signs": lambda: rng.standard_normal(N) * 10.0 ** rng.integers(-30, 30, N),
         "tenths": lambda: rng.integers(0, 10, N) / 10, "pairs": lambda: rng.permutation(np.arange(N) // 2).astype(float),
         "hundreds": lambda: np.exp(rng.integers(0, 1 + N // 100, N) / 7.0 % 40), "one value": lambda: np.full(N, 0.25),
         "infinities": lambda: np.where(rng.random(N) < 0.3, np.inf, rng.standard_normal(N)) * np.where(rng.random(N) < 0.3, -1, 1)}[kind]().astype(np.float32)
    score = torch.from_numpy(x).cuda()
    ctx = pb.Context(64, 1, 1, 64, torch.bfloat16, torch.float32)
    out = [torch.full((N,), 7, dtype=dt, device="cuda") for dt in (torch.uint8, torch.int32, torch.int32)] + [torch.zeros(2, dtype=torch.int32, device="cuda")]
    for lam in (0.0, 0.3, 0.5, 0.97, 1.0):
        ctx.pact_prune(score, pb.make_params(lam=lam), *out)
        _, keep, kept, pruned = orc.split(x, lam)
        assert out[3].cpu().tolist() == [kept.size, pruned.size]
        assert np.array_equal(out[0].cpu().numpy().astype(bool), keep)
        assert np.array_equal(out[1][:kept.size].cpu().numpy(), kept) and np.array_equal(out[2][:pruned.size].cpu().numpy(), pruned)


@pytest.mark.parametrize("case", ["many rows", "more survivors than estimated"])
def test_centres_outside_shared_memory(case):
    """Blocks of more than 1024 rows, adjacency words and densities that stay in global memory."""
    if case == "many rows":                   # sixteen images, so nine CTAs for the large one
        wls = [_workload(9400 if b == 3 else 5 + b, 1, 1, 8, 8, torch.bfloat16, 40 + b) for b in range(16)]
        wl = workloads.Workload("edge", [w.images[0] for w in wls], 8, 1, 1, 8, torch.bfloat16, 0.0, 0.3)
    else:                                     # six groups of equal scores; the threshold is in one of them
        wl = _workload(1800, 4, 2, 64, 256, torch.bfloat16, 3)
        img, pick = wl.images[0], torch.arange(1800) % 6
        img.K.copy_(img.K[pick]); img.Q.copy_(img.Q[pick]); img.H[1:1801] = img.H[1:1801][pick]
    _check(wl, torch.float32)


def test_centres_left_open_are_resolved():
    """Rows that the sweeps give up on are resolved by the kernel that lists the centres."""
    from paper_2504_08966_b200 import binding as pb
    wl = workloads.single_image(seed=29, N=2000, T=8, n_blobs=50)
    img = wl.images[0]
    ctx = pb.Context(wl.d, wl.n_qh, wl.n_kvh, wl.d_h, wl.dtype, torch.float32)
    im = pb.device_image(img, torch.float32)
    ctx.set_wait_limits(center_sweeps=1)
    ctx.pact_reduce([im], pb.make_params(lam=wl.lam, d_c=wl.d_c, d_n=wl.d_n, alpha=wl.alpha))
    torch.cuda.synchronize()
    assert int(im.counters[pb.CNT["status"]]) == -5
    assert np.array_equal(im.label.cpu().numpy(), oracle_image(wl, img)["label"])


@pytest.mark.parametrize("N,T,vis,d,rope,pinned", [
    (3, 0, 0, 64, False, True),               # smaller than the parts
    (780, 9, 2, 8192, False, True),           # just above the size that arrives in parts, one-cluster step
    (760, 0, 0, 8192, True, True),            # just below it
    (2309, 40, 40, 3584, True, True), (2309, 40, 0, 3584, False, False), (700, 5, 1, 64, False, False),
])
def test_host_buffers(N, T, vis, d, rope, pinned):
    """Inputs in parts or not, results written to host memory by the kernels or copied."""
    from paper_2504_08966_b200 import binding as pb
    wl = _workload(N, 4, 2, 64, d, torch.bfloat16, N + T, rope=rope, T=T)
    img = wl.images[0]
    img.vis_start = vis
    ctx = pb.Context(wl.d, wl.n_qh, wl.n_kvh, wl.d_h, wl.dtype, torch.float32)
    z = lambda m, dt: torch.full(m, 7, dtype=dt).pin_memory() if pinned else torch.full(m, 7, dtype=dt)   # noqa: E731
    n = N + T
    host = dict(H=img.H.pin_memory(), K_euti=img.K.pin_memory(), Q_euti=img.Q.pin_memory(), P=img.P.pin_memory(), vis_start=vis, N=N)
    results = dict(H_out=z((n, d), torch.float32), P_out=z((n,), torch.int32), size_out=z((n,), torch.int32), logw_out=z((n,), torch.float32),
                   label=z((N,), torch.int32), counters=z((16,), torch.int32))
    host.update(results)
    host["K_clu"] = img.K_clu.pin_memory() if rope else host["K_euti"]
    staging = torch.empty(ctx.host_staging_bytes(n, N), dtype=torch.uint8, device="cuda")
    want = gpu_reduce(wl, torch.float32)[0][0]
    for _ in range(3):                        # (large hidden states come in parts from the second call on)
        for t in results.values():
            t.fill_(7)
        staging.fill_(255)                    # nothing of the call before is left to be found
        ctx.pact_reduce_host(host, pb.make_params(lam=wl.lam, d_c=wl.d_c), staging)
        _same_as_device(host, want)
        n_out = want["n_out"]
        assert bool((host["H_out"][n_out:] == 7).all()) and bool((host["P_out"][n_out:] == 7).all())


def _host_call(wl, ctx, params=None):
    """pact_reduce_host on pinned copies of the workload's image; the staging buffer holds nothing of an earlier call."""
    from paper_2504_08966_b200 import binding as pb
    img, n = wl.images[0], wl.images[0].n_total
    z = lambda m, dt: torch.full(m, 7, dtype=dt).pin_memory()   # noqa: E731
    host = dict(H=img.H.pin_memory(), K_euti=img.K.pin_memory(), Q_euti=img.Q.pin_memory(), P=img.P.pin_memory(), vis_start=img.vis_start, N=img.N,
                H_out=z((n, wl.d), ctx.out_dtype), P_out=z((n,), torch.int32), size_out=z((n,), torch.int32), logw_out=z((n,), torch.float32),
                label=z((img.N,), torch.int32), counters=z((16,), torch.int32))
    host["K_clu"] = host["K_euti"]
    staging = torch.full((ctx.host_staging_bytes(n, img.N),), 255, dtype=torch.uint8, device="cuda")
    ctx.pact_reduce_host(host, params or pb.make_params(lam=wl.lam, d_c=wl.d_c), staging)
    return host


def _same_as_device(host, want):
    n_out = int(host["counters"][0])
    assert int(host["counters"][8]) == 0 and n_out == want["n_out"] and np.array_equal(host["label"].numpy(), want["label"])
    for key in ("P_out", "size_out", "logw_out"):
        assert np.array_equal(host[key][:n_out].numpy(), want[key])
    assert torch.equal(host["H_out"][:n_out], want["H_out_raw"])


@pytest.mark.parametrize("N", [1, 3, 7, 8, 9])
def test_host_buffers_of_a_tiny_image_in_a_long_prompt(N):
    """The part of the hidden states that holds no visual token still holds the text behind the image: 13 MB of it."""
    from paper_2504_08966_b200 import binding as pb
    wl = _workload(N, 4, 2, 64, 3584, torch.bfloat16, N, T=1850)
    ctx = pb.Context(wl.d, wl.n_qh, wl.n_kvh, wl.d_h, wl.dtype, torch.float32)
    want = gpu_reduce(wl, torch.float32)[0][0]
    for _ in range(3):
        _same_as_device(_host_call(wl, ctx), want)


def test_no_norm_and_norm_only():
    """Both forms of the score without one of its factors, over several units of the token pass."""
    from paper_2504_08966_b200 import binding as pb
    wl = _workload(5000, 4, 2, 64, 256, torch.bfloat16, 5)
    for flags, kw in ((pb.FLAG_NO_NORM, {"use_norm": False}), (pb.FLAG_NORM_ONLY, {"use_query": False})):
        outs, _ = gpu_reduce(wl, torch.float32, params=pb.make_params(lam=0.5, d_c=0.3, flags=flags))
        assert not compare_image(oracle_image(wl, wl.images[0], **kw), outs[0], wl.images[0], False)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("N,n_qh,n_kvh,d_h", [(5, 1, 1, 8), (300, 4, 2, 64), (1500, 7, 1, 40), (5000, 4, 4, 128)])
def test_non_finite_queries_and_keys_reach_the_scores(N, n_qh, n_kvh, d_h, dtype):
    """An infinity or a NaN in the queries or the scoring keys makes every score NaN."""
    from paper_2504_08966_b200 import binding as pb
    wl = _workload(N, n_qh, n_kvh, d_h, 64, dtype, 5 * N, rope=True)
    img = wl.images[0]
    ctx = pb.Context(wl.d, n_qh, n_kvh, d_h, dtype, torch.float32)
    col = n_kvh * d_h - 1                     # last element of the last head
    for what in ("Q", "K"):
        for value in (np.nan, np.inf, -np.inf):
            t = getattr(img, what)
            old = t[N - 2, col].clone()
            t[N - 2, col] = value
            im = pb.device_image(img, torch.float32)
            t[N - 2, col] = old
            score = torch.zeros(N, dtype=torch.float32, device="cuda")
            ctx.pact_importance(im, pb.make_params(), score)
            assert bool(score.isnan().all()), (what, value)
            if N > 100:                       # and the whole step: every token shares the threshold, so all survive
                ctx.pact_reduce([im], pb.make_params())
                torch.cuda.synchronize()
                assert bool(im.score.isnan().all()) and int(im.counters[pb.CNT["q"]]) == N and int(im.counters[pb.CNT["status"]]) == 0


@pytest.mark.parametrize("n_qh,n_kvh,d_h,d,dtype", [
    (1, 1, 26496, 8192, torch.bfloat16),      # the last width whose query fits beside the smallest row buffers
    (1, 1, 26504, 8192, torch.bfloat16), (1, 1, 28896, 64, torch.bfloat16), (32, 1, 872, 3584, torch.bfloat16), (1, 1, 28896, 2056, torch.float32),
])
def test_widest_queries(n_qh, n_kvh, d_h, d, dtype):
    """Queries that leave little or no shared memory to the token pass; 28928 columns less 32 per head are the most that are taken."""
    from paper_2504_08966_b200 import binding as pb
    N = 43
    g = torch.Generator().manual_seed(d_h)
    t = lambda m, n: (0.1 * torch.randn(m, n, generator=g)).to(dtype)   # noqa: E731
    img = workloads.Image(H=t(N, d), K=t(N, n_kvh * d_h), Q=t(N, n_qh * d_h), P=torch.arange(N, dtype=torch.int32), n_total=N, vis_start=0, N=N)
    wl = workloads.Workload("wide", [img], d, n_qh, n_kvh, d_h, dtype, 0.5, 0.3)
    _check(wl, torch.float32)
    with pytest.raises(pb.PactError):
        pb.Context(64, 1, 1, 28904, dtype, torch.float32)


@pytest.mark.parametrize("N,limit", [(600, 0), (2601, 0), (600, 1)])
def test_a_chain_of_centres(N, limit):
    """Row k is a neighbour of rows k - 1 and k + 1 only and all densities but the ends' are equal: rows 1, 3, 5, ... become
    centres one after the other, more of them than the sweeps a CTA may spend without seeing progress."""
    from paper_2504_08966_b200 import binding as pb
    d_k = (N + 64) // 64 * 64
    i = torch.arange(N, device="cuda")
    K = torch.zeros(N, d_k, dtype=torch.bfloat16, device="cuda")
    K[i, i] = 1
    K[i, i + 1] = 1                           # neighbours at distance 1/2, all others at 1
    ctx = pb.Context(64, 1, 1, d_k, torch.bfloat16, torch.float32)
    ctx.set_wait_limits(center_sweeps=limit)
    z = lambda n, dt=torch.int32: torch.zeros(n, dtype=dt, device="cuda")   # noqa: E731
    cidx, C, label, cnt = z(N), z(1), z(N), z(16)
    ctx.pact_dbdpc(K, i.int(), torch.tensor([N], dtype=torch.int32, device="cuda"), pb.make_params(lam=0.0, d_c=0.75), z(N, torch.float32), cidx, C, label, cnt)
    want = list(range(1, N - 1, 2)) + ([N - 1] if N % 2 == 0 else [])     # an end's density is the smallest
    assert cidx[:int(C)].tolist() == want
    assert label.tolist() == [max(0, (k - 1) // 2) for k in range(N)]
    assert int(cnt[pb.CNT["status"]]) == (-5 if limit else 0)
    assert int(cnt[pb.CNT["sweeps"]]) > (512 if N > 2000 else 1)


@pytest.mark.parametrize("N,n_kvh,d_h,dtype,lam,B,kernels", [
    (256, 4, 128, torch.float32, 0.5, 1, 4), (256, 4, 128, torch.float32, 0.0, 1, 10), (128, 8, 128, torch.float32, 0.0, 1, 4),
    (640, 4, 128, torch.float32, 0.0, 1, 10), (300, 5, 104, torch.bfloat16, 0.0, 1, 10), (512, 1, 64, torch.float32, 0.5, 2, 4),
    (512, 1, 64, torch.bfloat16, 0.0, 1, 4), (513, 1, 64, torch.bfloat16, 0.0, 1, 10), (1024, 1, 64, torch.bfloat16, 0.5, 2, 4),
    (777, 8, 128, torch.bfloat16, 0.5, 1, 4), (778, 8, 128, torch.bfloat16, 0.5, 1, 10),
])
def test_one_cluster_or_the_whole_gpu(N, n_kvh, d_h, dtype, lam, B, kernels):
    """Both sides of the lines between the one-cluster step and the wide kernels: survivors, key width, images."""
    wls = [_workload(N - b, n_kvh, n_kvh, d_h, 64, dtype, 3 * N + b) for b in range(B)]
    wl = workloads.Workload("line", [w.images[0] for w in wls], 64, n_kvh, n_kvh, d_h, dtype, lam, 0.3)
    outs, ctx = gpu_reduce(wl, torch.float32)
    assert ctx.launch_count() == kernels
    for img, g in zip(wl.images, outs):
        o = oracle_image(wl, img)
        bad = compare_image(o, g, img, False)
        assert not bad, f"{bad}; fragile: {fragile_report(o, wl.d_c, wl.alpha)}"


def test_first_host_call_of_a_context_needs_no_stream_of_its_own():
    """Hidden states arrive in parts from the second call on (a kernel more for each part)."""
    from paper_2504_08966_b200 import binding as pb
    wl = _workload(900, 2, 2, 64, 8192, torch.bfloat16, 17)
    ctx = pb.Context(wl.d, wl.n_qh, wl.n_kvh, wl.d_h, wl.dtype, torch.float32)
    want = gpu_reduce(wl, torch.float32)[0][0]
    counts = [0]
    for _ in range(3):
        _same_as_device(_host_call(wl, ctx), want)
        counts.append(ctx.launch_count())
    assert np.diff(counts).tolist() == [4, 6, 6]


@pytest.mark.parametrize("N,T,d", [(2309, 40, 3584), (900, 3, 8192)])
def test_host_buffers_with_the_flags_of_the_ablations(N, T, d):
    """Hidden states in parts, with the score's factors left out and with centres in place of means: the wide kernels and the
    one-cluster step."""
    from paper_2504_08966_b200 import binding as pb
    wl = _workload(N, 4, 2, 64, d, torch.bfloat16, N + 1, T=T)
    for flags in (pb.FLAG_NO_NORM, pb.FLAG_NORM_ONLY, pb.FLAG_CENTER_ONLY, pb.FLAG_CENTER_ONLY | pb.FLAG_NO_NORM):
        params = pb.make_params(lam=wl.lam, d_c=wl.d_c, flags=flags)
        want = gpu_reduce(wl, torch.float32, params=params)[0][0]
        ctx = pb.Context(wl.d, wl.n_qh, wl.n_kvh, wl.d_h, wl.dtype, torch.float32)
        for _ in range(3):
            _same_as_device(_host_call(wl, ctx, params), want)


def test_merged_rows_of_any_bf16_value():
    """Rows with every bf16 value (subnormal numbers, infinities, NaN): text rows and clusters of one row, and sums of two in fp32."""
    from paper_2504_08966_b200 import binding as pb
    d, N, T = 4096, 18, 14
    bits = torch.arange(65536, dtype=torch.int32).reshape(16, d).to(torch.int16).view(torch.bfloat16)
    H = torch.cat([bits, bits]).cuda()                # token i of the second half of the rows is row i + T
    z = lambda m, dt: torch.zeros(m, dtype=dt, device="cuda")   # noqa: E731
    K = z((N, 64), torch.bfloat16)
    label = torch.arange(N, dtype=torch.int32, device="cuda") % 17           # tokens 0 and 17 share a cluster
    im = pb.DeviceImage(H, K, K, K, torch.arange(N + T, dtype=torch.int32, device="cuda"), T, N, z((N + T, d), torch.float32), z(N + T, torch.int32),
                        z(N + T, torch.int32), z(N, torch.int32), z(N, torch.float32), z(N, torch.uint8), z(pb.N_COUNTERS, torch.int32))
    pb.Context(d, 1, 1, 64, torch.bfloat16, torch.float32).pact_merge(im, label, torch.arange(17, dtype=torch.int32, device="cuda"),
                                                                      torch.tensor([17], dtype=torch.int32, device="cuda"), pb.make_params())
    want = 0.0 + H[:T + 17].float()                   # (a sum begins at +0)
    want[T] = (want[T] + H[T + 17].float()) * 0.5
    got = im.H_out[:T + 17]
    assert torch.equal(torch.isnan(got), torch.isnan(want))
    assert torch.equal(torch.nan_to_num(got, nan=0.0).view(torch.int32), torch.nan_to_num(want, nan=0.0).view(torch.int32))


@pytest.mark.parametrize("C", [1, 31, 33, 257, 500, 513, 1030])
@pytest.mark.parametrize("N,n_kvh,d_h", [(1100, 1, 64), (3000, 3, 64), (7290, 4, 128), (19100, 2, 64)])
def test_nearest_centres_in_tiles(N, n_kvh, d_h, C):
    """Rows x centres at the edges of its tiles: one round of equal tiles (up to 512 centres wide) and rounds of 256, one K-slab per stage and two."""
    from paper_2504_08966_b200 import binding as pb
    g = torch.Generator(device="cuda").manual_seed(N + C)
    K = torch.randn(N, n_kvh * d_h, device="cuda", generator=g).to(torch.bfloat16)
    i32 = lambda x: torch.as_tensor(x, dtype=torch.int32, device="cuda")   # noqa: E731
    cen = torch.randperm(N, device="cuda", generator=g)[:C].sort().values
    rows = torch.ones(N, dtype=torch.bool, device="cuda")
    rows[cen] = False
    pruned = rows.nonzero().flatten()
    label, r = torch.full((N,), -7, dtype=torch.int32, device="cuda"), i32([0])
    ctx = pb.Context(256, n_kvh, n_kvh, d_h)
    ctx.pact_reincorporate(K, i32(pruned), i32([pruned.numel()]), i32(cen), i32([C]), pb.make_params(d_c=2.0, alpha=1.5), label, r)
    assert int(r) == pruned.numel() and bool((label[cen] == -7).all())
    Kd = torch.nn.functional.normalize(K.double(), dim=1)
    dist = 1.0 - Kd[pruned] @ Kd[cen].T
    got = label[pruned].long()
    assert int(got.min()) >= 0 and int(got.max()) < C
    # a dot product of d_k terms in fp32 is good to about 1e-6 of the norms
    assert float((dist.gather(1, got[:, None])[:, 0] - dist.min(1).values).max()) < 2e-6


@pytest.mark.parametrize("N,C,d", [(9, 2, 3584), (41, 3, 3584), (57, 2, 896), (95, 1, 1024), (97, 30, 896), (600, 11, 3584), (881, 25, 896), (1200, 36, 3584)])
def test_merge_ranges_of_few_rows(N, C, d):
    """Ranges of eight and twelve items, clusters that end up to 24 items past theirs and clusters cut at every boundary."""
    test_merge_ranges(N, C, 5, d, torch.bfloat16)
