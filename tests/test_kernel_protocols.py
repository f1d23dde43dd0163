"""Rules that the kernels' sources have to keep so that no CTA can wait for ever, checked by reading the sources: what they
guard against cannot be provoked on a GPU without hanging it.

A device-side wait on an mbarrier or a counter is bounded, and the bound runs out for each thread by itself: of two threads
at the same wait one may give up while the other finds it complete.  A barrier of many threads has no bound.  So whether a
thread arrives at one must not depend on how a bounded wait ended."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(__file__)), "paper_2602_03681_b200", "csrc")
SOURCES = sorted(os.path.basename(p) for p in glob.glob(os.path.join(CSRC, "*.cu")))
BARRIER = re.compile(r"\b(named_barrier_sync|__syncthreads\w*)\s*\(")
WAIT = r"\b(?:mbar_wait|wait_all|wait_counter_ge)\s*\("


def kernels(path):
    """[(name, body without comments)] of a source file."""
    with open(path) as f:
        text = f.read()
    text = re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))
    found = []
    for m in re.finditer(r"__global__[^;{]*?\b(\w+_kernel)\(", text):
        at = text.index("{", m.end())
        depth, end = 1, at + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[end], 0)
            end += 1
        found.append((m.group(1), text[at + 1:end - 1]))
    return found


def barriers_behind_a_wait(body):
    """The barriers of a kernel that a thread may miss because of how its own bounded wait ended: under a condition on the
    outcome, or in what a break, continue or return under such a condition leaves (continue: the rest of the block around it)."""
    outcomes = set(re.findall(r"(\w+)\s*=[^=;{}]*" + WAIT, body))
    while True:      # (variables set from those)
        more = set(re.findall(r"(\w+)\s*=[^=;{}]*\b(?:%s)\b" % "|".join(outcomes), body)) if outcomes else set()
        if more <= outcomes:
            break
        outcomes |= more
    decided = re.compile(WAIT + "".join(r"|\b%s\b" % n for n in sorted(outcomes)))
    missed, stack, start, i = [], [], 0, 0
    while i < len(body):
        ch = body[i]
        if ch == "(":                                         # (a for header's semicolons end no statement)
            depth = 1
            while depth:
                i += 1
                depth += {"(": 1, ")": -1}.get(body[i], 0)
        if ch in "{;}":
            words = body[start:i]
            cond = bool(re.search(r"\b(if|while|for)\s*\(", words)) and bool(decided.search(words))
            if BARRIER.search(words) and "mbar_" not in words:
                block = next((b for b in reversed(stack) if b["left"] or b["cond"]), None)
                if cond or block:
                    missed.append(" ".join(words.split()))
                for b in stack:
                    b["barriers"].append(" ".join(words.split()))
            leave = re.search(r"\b(break|continue|return)\b", words)
            if leave and (cond or any(b["cond"] for b in stack)):
                for b in reversed(stack):
                    if b["function"]:                         # (a lambda's own return)
                        break
                    if leave.group(1) != "return" and b["loop"]:
                        if leave.group(1) == "break":         # (the loop's next turn, too, is missed)
                            missed += b["barriers"]
                            b["cond"] = True
                        elif not b["cond"]:
                            around = [x for x in stack[stack.index(b):] if not x["cond"]]
                            around[-1]["left"] = True
                        break
                    if leave.group(1) == "return":
                        b["left"] = True
            if ch == "{":
                stack.append(dict(cond=cond, loop=bool(re.search(r"\b(for|while)\s*\(|\bdo$", words.strip())),
                                  function=bool(re.search(r"\]\s*(\(.*\))?\s*(->.*)?$", words, re.S)), left=False, barriers=[]))
            elif ch == "}" and stack:
                stack.pop()
            start = i + 1
        i += 1
    return missed


@pytest.mark.parametrize("source", SOURCES)
def test_no_barrier_stands_behind_one_threads_wait(source):
    for name, body in kernels(os.path.join(CSRC, source)):
        assert not barriers_behind_a_wait(body), name


def lets_dependents_in_too_early(body):
    """Whether a kernel that allocates tensor memory may let a programmatic dependent start before every CTA has its
    columns: the dependent may hold columns while it waits for this kernel, and an allocation waits without a limit."""
    alloc, release = body.find("tmem_alloc("), body.find("launch_dependents()")
    if alloc < 0 or release < 0:
        return False
    if re.search(r"\{\s*tmem_alloc\([^;]*;\s*launch_dependents\(\)", body):       # (the allocating warp itself)
        return body.count("launch_dependents()") != 1
    barrier = BARRIER.search(body, alloc)
    return barrier is None or release < barrier.end()


@pytest.mark.parametrize("source", SOURCES)
def test_dependents_start_behind_the_allocation_of_tensor_memory(source):
    for name, body in kernels(os.path.join(CSRC, source)):
        assert not lets_dependents_in_too_early(body), name


def test_the_rules_find_what_they_are_for():
    assert lets_dependents_in_too_early("launch_dependents(); if (w) tmem_alloc(&b, 64); __syncthreads();")
    assert lets_dependents_in_too_early("if (w) tmem_alloc(&b, 64); launch_dependents(); __syncthreads();")
    assert lets_dependents_in_too_early("launch_dependents(); if (w) { tmem_alloc(&b, 64); launch_dependents(); }")
    assert not lets_dependents_in_too_early("if (w) tmem_alloc(&b, 64); __syncthreads(); launch_dependents();")
    assert not lets_dependents_in_too_early("if (w) { tmem_alloc(&b, 64); launch_dependents(); } __syncthreads();")
    ok = "bool ok = mbar_wait(&a, 0, f); "
    assert barriers_behind_a_wait(ok + "if (ok) { x(); if (y) { named_barrier_sync(1, 64); } }")
    assert barriers_behind_a_wait(ok + "if (ok) __syncthreads();")
    assert barriers_behind_a_wait("for (int t = 0; t < T; ++t) { __syncthreads(); if (!mbar_wait(&a, 0, f)) break; }")
    assert barriers_behind_a_wait("for (int t = 0; t < T; ++t) { if (!mbar_wait(&a, 0, f)) continue; __syncthreads(); }")
    assert barriers_behind_a_wait("for (int t = 0; t < T; ++t) { if (!mbar_wait(&a, 0, f)) { --n; continue; } __syncthreads(); }")
    assert barriers_behind_a_wait("bool ok = true; for (int t = 0; ok && t < T; ++t) { __syncthreads(); ok = mbar_wait(&a, 0, f); }")
    assert not barriers_behind_a_wait(ok + "if (ok) { x(); } __syncthreads();")
    assert not barriers_behind_a_wait("for (;;) { if (p) { if (!mbar_wait(&a, 0, f)) continue; } else { __syncthreads(); } }")
    assert not barriers_behind_a_wait("for (;;) { for (;;) { if (!mbar_wait(&a, 0, f)) break; } __syncthreads(); }")
