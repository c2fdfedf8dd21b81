"""Pairs of CTAs (all pairs and rows x centres of batches, largest key distance) on several streams at once, beside single CTAs with tensor
memory.  In a process of its own that looks at events until a deadline, so that a call without end is a failure and not a wait."""
import os
import subprocess
import sys
import time

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _images(pb, torch, seed, B, N, d):
    g = torch.Generator(device="cuda").manual_seed(seed)
    rand = lambda *s: torch.randn(*s, device="cuda", generator=g)   # noqa: E731
    z = lambda m, dt: torch.zeros(m, dtype=dt, device="cuda")   # noqa: E731
    out = []
    for _ in range(B):
        K = (rand(N // 8, 64)[torch.randint(0, N // 8, (N,), device="cuda", generator=g)] + 0.2 * rand(N, 64)).to(torch.bfloat16)
        out.append(pb.DeviceImage(rand(N, d).to(torch.bfloat16), K, rand(N, 64).to(torch.bfloat16), K, torch.arange(N, dtype=torch.int32, device="cuda"), 0, N,
                                  z((N, d), torch.float32), z(N, torch.int32), z(N, torch.int32), z(N, torch.int32), z(N, torch.float32), z(N, torch.uint8),
                                  z(pb.N_COUNTERS, torch.int32), z(N, torch.float32)))
    return out


def _child(rounds, deadline):
    sys.path.insert(0, ROOT)
    import torch
    from paper_2504_08966_b200 import binding as pb
    params = pb.make_params(lam=0.4, d_c=0.2)
    calls, status = [], []                                  # (call, its outputs), one for each stream
    # 16 x 2600 tokens: 13 x 14 / 2 blocks of survivors per image and 21 x 16 row blocks, both passes on pairs; 1800 tokens: single CTAs
    for B, N in ((16, 2600), (16, 2600), (1, 1800)):
        ctx, ims = pb.Context(64, 1, 1, 64, torch.bfloat16, torch.float32), _images(pb, torch, len(calls), B, N, 64)
        ctx.ensure_workspace(B, N)
        calls.append((lambda ctx=ctx, ims=ims: ctx.pact_reduce(ims, params), [t for im in ims for t in (im.H_out, im.P_out, im.size_out, im.label, im.counters[:5])]))
        status += [im.counters[pb.CNT["status"]] for im in ims]
    layers = [im.K_clu for im in _images(pb, torch, 9, 10, 2600, 64)]
    md, lo, ctx = torch.zeros(10, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda"), pb.Context(64, 1, 1, 64, torch.bfloat16, torch.float32)
    calls.append((lambda: ctx.pact_key_spread(layers, 0.3, md, lo), [md, lo]))

    def wait(streams):
        events, end = [s.record_event() for s in streams], time.monotonic() + deadline
        while not all(e.query() for e in events):
            if time.monotonic() > end:
                os.write(2, f"streams at their end: {[e.query() for e in events]}\n".encode())
                os._exit(3)                                 # (no destructor would come back either)
            time.sleep(0.001)

    def forget():
        for _, outs in calls:
            for t in outs:
                t.fill_(7)

    alone = []
    forget()
    for call, outs in calls:
        call()
        wait([torch.cuda.current_stream()])
        alone.append([t.clone() for t in outs])
    forget()
    wait([torch.cuda.current_stream()])
    streams = [torch.cuda.Stream() for _ in calls]
    for r in range(rounds):
        for s, (call, _) in zip(streams, calls):
            with torch.cuda.stream(s):
                call()
        if r % 8 == 7:
            wait(streams)
    wait(streams)
    for (_, outs), want in zip(calls, alone):
        for t, w in zip(outs, want):
            if not torch.equal(t, w):
                os.write(2, b"not what the call gives alone\n")
                os._exit(4)
    assert all(int(x) == 0 for x in status)
    print("all streams ended")


@pytest.mark.gpu
def test_pairs_of_ctas_on_several_streams_end():
    r = subprocess.run([sys.executable, os.path.abspath(__file__), "64", "20"], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "all streams ended" in r.stdout, r.stderr[-2000:]


if __name__ == "__main__":
    _child(int(sys.argv[1]), float(sys.argv[2]))
