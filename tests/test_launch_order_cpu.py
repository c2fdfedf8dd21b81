"""Kernels read ahead of pdl_wait() what comes from before their predecessor (csrc/common.cuh).  That rests on every kernel of
the chain: no trigger and no return before the wait.  Read from the source, block by block."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2504_08966_b200", "csrc")
FILES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))


def _read(name):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    return re.sub(r"/\*.*?\*/", "", text, flags=re.S)


def _kernels(text):
    """(name, body) of every __global__ function."""
    for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\(", text):
        start = text.index("{", m.end())
        depth, i = 1, start + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(1), text[start:i]


def _too_early(body):
    """Triggers and returns that no wait precedes in their block or one around it (returns of lambdas aside)."""
    waited, in_lambda, bad, begin = [False], [False], [], 0
    for m in re.finditer(r"[{};]|\bpdl_wait\(\)|\bpdl_trigger\(\)|\breturn\b", body):
        tok = m.group(0)
        if tok == "{":
            waited.append(waited[-1])
            in_lambda.append(in_lambda[-1] or bool(re.search(r"\[&?\]\s*\(", body[begin:m.start()])))
        elif tok == "}":
            waited.pop()
            in_lambda.pop()
        elif tok == "pdl_wait()":
            waited[-1] = True
        elif tok == "pdl_trigger()" and not waited[-1]:
            bad.append("trigger")
        elif tok == "return" and not waited[-1] and not in_lambda[-1]:
            bad.append("return")
        if tok in "{};":
            begin = m.end()
    return bad


KERNELS = [(f, name, body) for f in FILES for name, body in _kernels(_read(f))]


def test_all_kernels_are_found():
    names = {name for _, name, _ in KERNELS}
    assert {"k_qsum", "k_tokens", "k_scores", "k_select", "k_split", "k_split_regs", "k_tiles_umma", "k_tiles_pair", "k_centers", "k_center_keys", "k_members",
            "k_lists", "k_merge", "k_small"} <= names


@pytest.mark.parametrize("f,name,body", [pytest.param(*k, id=k[1]) for k in KERNELS])
def test_nothing_is_triggered_before_the_wait(f, name, body):
    assert "pdl_wait()" in body and not _too_early(body), f


def test_a_planted_trigger_is_found():
    for name, want in (("k_select", ["trigger"]), ("k_qsum", ["trigger"]), ("k_centers", ["trigger"])):
        body = next(b for _, n, b in KERNELS if n == name)
        early = re.sub(r"pdl_wait\(\);\s*pdl_trigger\(\);", "pdl_trigger(); pdl_wait();", body, count=1)
        assert early != body and _too_early(early) == want
    body = next(b for _, n, b in KERNELS if n == "k_scores")
    assert _too_early(body.replace("pdl_wait();", ";", 1)) == ["return"]


def _headers(body, at):
    """The statement at this place from its start, and the head of every block around it."""
    heads, i = [body[max(body.rfind(c, 0, at) for c in "{};") + 1:at]], at
    while True:
        depth, i = 0, i - 1
        while i >= 0 and (depth or body[i] != "{"):
            depth += {"}": 1, "{": -1}.get(body[i], 0)
            i -= 1
        if i < 0:
            return heads
        begin = i                                          # a head ends at its brace and may hold the semicolons of a for
        depth = 0
        while begin > 0 and (depth or body[begin - 1] not in "{};"):
            begin -= 1
            depth += {")": 1, "(": -1}.get(body[begin], 0)
        heads.append(body[begin:i])


def _not_asked_for(body, call, bit):
    """Calls of `call` that are reached in a launch without the part `bit` of the token pass."""
    return [m.start() for m in re.finditer(re.escape(call), body) if not any(f"what & {bit}" in h for h in _headers(body, m.start()))]


def test_the_token_pass_asks_for_no_copies_that_it_does_not_wait_for():
    """A launch without norms (or without logits) has no wait for rows (or keys)."""
    body = next(b for _, n, b in KERNELS if n == "k_tokens")
    for call, wait, bit in (("issue_row();", "mbar_wait_warp(&s_rbar", "kTokNorms"), ("issue_keys(u0", "mbar_wait_warp_unless(&s_abort, &s_kbar", "kTokLogits"), ("issue_keys(mu", "mbar_wait_warp_unless(&s_abort, &s_kbar", "kTokLogits")):
        assert call in body and wait in body
        assert not _not_asked_for(body, call, bit), call
        assert not _not_asked_for(body, wait, bit), wait
    bare = body.replace("if (lane == 0 && (what & kTokNorms)) issue_row();", "if (lane == 0) issue_row();")
    assert bare != body and len(_not_asked_for(bare, "issue_row();", "kTokNorms")) == 1


def _pair_steps(body):
    """Barriers of the whole cluster, collective allocations and deallocations of a pair's tensor memory and returns, in order; those inside a
    block, i.e. not on every way through the kernel, in brackets (returns of lambdas aside)."""
    depth, steps = -1, []                                  # (the body's own brace comes first)
    for m in re.finditer(r"[{}]|\bcluster_(?:barrier|arrive|wait)\(\)|\btmem_alloc2\(|\btmem_dealloc2\(|\breturn\b", body):
        tok = m.group(0).rstrip("()")
        depth += {"{": 1, "}": -1}.get(tok, 0)
        if tok not in "{}" and (depth == 0 or tok != "return"):
            steps.append(f"[{tok}]" if depth else tok)
    return steps


def test_pairs_of_ctas_ask_for_tensor_memory_between_cluster_barriers():
    """A CTA may ask for tensor memory of its pair only once the other one runs, and leave only when both have theirs back."""
    pairs = [(n, b) for _, n, b in KERNELS if "tmem_alloc2(" in b]
    assert [n for n, _ in pairs] == ["k_tiles_pair"]
    want = ["cluster_arrive", "cluster_wait", "tmem_alloc2", "cluster_arrive", "cluster_wait", "cluster_barrier", "tmem_dealloc2", "cluster_barrier"]
    for _, body in pairs:
        assert _pair_steps(body) == want
        assert _pair_steps(body.replace("pdl_wait();", "if (rank) return; pdl_wait();", 1)) != want


def test_every_kernel_that_is_launched_is_found():
    """No kernel of the sources escapes the checks above, those least that read ahead of their wait."""
    declared = {m for f in FILES for m in re.findall(r"\b(?:launch_k|launch_opt|launch_coop)\(\s*(?:\w+,\s*)?(k_\w+)", _read(f))}
    assert {"k_assign", "k_label_counts", "k_list_clear"} <= {name for _, name, _ in KERNELS}
    assert len(declared) > 10 and declared <= {name for _, name, _ in KERNELS}
