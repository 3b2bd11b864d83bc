"""Orderings that a run rarely shows to be missing, checked on the text of the CUDA sources (CPU).

Asynchronous copies: cp.async.wait_group covers committed groups only: a copy that was issued and never committed is not ordered before what follows
the wait.  So each function or lambda that issues copies commits them, hands them to an mbarrier, or belongs to a function whose
only wait is cp_async_wait_all, which has to be cp.async.wait_all.

Tensor memory: a column pass follows a device-wide barrier, before which other warps read and multiplied into the words it
stores to.  tcgen05.fence::before_thread_sync stands before the barrier, so the pass opens with ::after_thread_sync."""
import os
import re

import pytest

from paper_2607_25234_gb300 import build

# helpers that issue copies for a caller that commits them or waits for all
ISSUERS = ("cp_async16", "cp_async16z", "cp_async16_zfill", "cp_async4", "copy16", "stage_block", "load_x_bf16")
ISSUE = re.compile(r"\b(?:%s)\s*(?:<\w+>)?\(|cp\.async\.c[ag]\.shared" % "|".join(ISSUERS))
WAIT_ALL = re.compile(r"cp_async_wait_all\(\)|cp\.async\.wait_all")
TRACKED = re.compile(r"cp_async_commit\(|cp\.async\.commit_group|cp_async_arrive\(")


def without_comments(text):
    return re.sub(r"//[^\n]*", "", text)


def body(text, brace):
    """The text from the opening brace to its match."""
    depth = 0
    for i in range(brace, len(text)):
        depth += (text[i] == "{") - (text[i] == "}")
        if depth == 0:
            return text[brace:i + 1]
    raise AssertionError("unbalanced braces")


def functions(text):
    """(name, body) of the device functions at namespace level."""
    text = re.sub(r"__launch_bounds__\((?:[^()]|\([^()]*\))*\)", "", text)
    for m in re.finditer(r"^[^\n;={}#]*\b(?:__device__|__global__)[^;{}]*?\b(\w+)\([^;{}]*\)[^;{}]*\{", text, re.M):
        yield m.group(1), body(text, m.end() - 1)


def lambdas(text):
    for m in re.finditer(r"\bauto (\w+) = \[[&=\w, ]*\](?:\([^()]*(?:\([^()]*\)[^()]*)*\))?\s*(?:mutable\s*)?\{", text):
        yield m.group(1), body(text, m.end() - 1)


def sources():
    return sorted(f for f in os.listdir(build.CSRC) if f.endswith((".cu", ".cuh")))


def read(name):
    with open(os.path.join(build.CSRC, name)) as f:
        return without_comments(f.read())


def test_wait_all_waits_for_uncommitted_copies_too():
    waits = dict(functions(read("whtmix_fast.cuh")))
    assert "cp.async.wait_all" in waits["cp_async_wait_all"] and "wait_group" not in waits["cp_async_wait_all"]


@pytest.mark.parametrize("name", sources())
def test_every_copy_is_committed_or_waited_for_with_the_rest(name):
    for fn, text in functions(read(name)):
        if fn in ISSUERS or not ISSUE.search(text):
            continue
        groups = "cp.async.wait_group" in text
        rest = text
        for lam, part in lambdas(text):
            rest = rest.replace(part, "")
            if lam not in ISSUERS and ISSUE.search(part):
                assert TRACKED.search(part) or (not groups and WAIT_ALL.search(text)), f"{name}: {fn}: {lam}"
        if ISSUE.search(rest):
            # (a lambda called afterwards may commit them with its own)
            assert TRACKED.search(text) or (not groups and WAIT_ALL.search(text)), f"{name}: {fn}"


def test_the_check_sees_a_missing_commit():
    kernel = '__device__ void f() { auto stage = [&](int g) { stage_block<64>(g); COMMIT }; stage(0); WAIT }'
    for commit, wait, ok in (("", 'asm("cp.async.wait_group 0;");', False), ("cp_async_commit();", 'asm("cp.async.wait_group 0;");', True),
                             ("", "cp_async_wait_all();", True)):
        (fn, text), = functions(kernel.replace("COMMIT", commit).replace("WAIT", wait))
        (lam, part), = lambdas(text)
        assert (fn, lam) == ("f", "stage") and ISSUE.search(part)
        assert bool(TRACKED.search(part) or ("cp.async.wait_group" not in text and WAIT_ALL.search(text))) == ok


@pytest.mark.parametrize("name", ["col_lanes", "col_regs_bwd", "col_lanes_bwd"])
def test_column_passes_open_with_the_tensor_memory_fence(name):
    text = dict(functions(read("whtmix_tri.cuh")))[name]
    stores = [m.start() for m in re.finditer(r"\bst_pairs<", text)]
    assert stores, "a pass through tensor memory"
    # the first statement loop over columns comes after the fence, whatever lambdas are defined before it
    loop = re.search(r"\n  for \(int g = ", text).start()
    assert loop < stores[0]
    opening = text[:loop]
    for _, part in lambdas(opening):
        opening = opening.replace(part, "")
    assert "tmem_fence_after()" in opening


def test_every_phase_that_touches_tensor_memory_ends_with_the_fence():
    fns = dict(functions(read("whtmix_tri.cuh")))
    assert fns["rows_in"].count("tmem_fence_before()") == 2  # each product's, and the end of the bf16 rows
    for name, calls in (("columns", 1), ("columns_bwd", 2)):
        assert fns[name].count("tmem_fence_before()") == calls, name
