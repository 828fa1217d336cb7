"""Kernels that are launched with programmatic serialization are resident while the kernel before them still writes what they
read.  The rule at launch() (csrc/common.cuh), checked in the sources: they wait before they touch global memory, and nothing they
run asks the compiler for non-coherent loads, which need data that stays unwritten for the whole life of the kernel and may be
moved above the wait."""
import functools
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_33135_b200", "csrc")
SOURCES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))


@functools.lru_cache(None)
def code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


@functools.lru_cache(None)
def bodies(text):
    """Function name -> (parameters, body), for functions defined at any depth; template instances share a name."""
    found = {}
    for m in re.finditer(r"\b(\w+)\s*\(", text):
        if m.group(1) in ("if", "for", "while", "switch", "asm", "sizeof", "defined", "__launch_bounds__"):
            continue
        i, depth = m.end(), 1
        while depth and i < len(text):
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        rest = re.match(r"\s*(const\s*)?\{", text[i:])
        if not rest:
            continue
        j, depth = i + rest.end(), 1
        while depth and j < len(text):
            depth += {"{": 1, "}": -1}.get(text[j], 0)
            j += 1
        p, b = found.get(m.group(1), ("", ""))
        found[m.group(1)] = (p + text[m.end():i], b + text[i:j])
    return found


@functools.lru_cache(None)
def launched():
    """Kernels that launch() or start() is given."""
    names = set()
    for f in SOURCES:
        for m in re.finditer(r"\b(?:launch|start)\s*(?:<([^;]*?)>)?\s*\(([^;]*);|\bkern = (\w+)", code(f)):
            names |= set(re.findall(r"\b\w+_kernel\b", " ".join(g for g in m.groups() if g)))
    return names


def test_the_rule_covers_the_kernels():
    assert {"colstat_kernel", "stat_fold_kernel", "quantize_tile_kernel", "quantize_token_kernel", "quantize_v_tile_kernel", "write_kv_kernel",
            "append_kv_kernel", "decode_prep_kernel", "decode_split_kernel", "decode_merge_kernel", "prefill_kernel"} <= launched()


@pytest.mark.parametrize("source", [f for f in SOURCES if f.endswith(".cu")])
def test_launched_kernels_wait_and_read_coherently(source):
    text = "".join(code(f) for f in SOURCES if f.endswith(".cuh")) + code(source)
    funcs = bodies(text)
    kernels = [k for k in funcs if k in launched()]
    for kernel in kernels:
        todo, seen = [kernel], set()
        while todo:                       # the kernel and every function of the library that it can reach
            f = todo.pop()
            if f in seen or f not in funcs:
                continue
            seen.add(f)
            params, body = funcs[f]
            assert not re.search(r"__ldg|\.nc\b|__ldc[gs]|__restrict__", params + body), (kernel, f)
            todo += re.findall(r"\b(\w+)\s*(?:<[^;{}()]*>)?\s*\(", body)
        body = funcs[kernel][1]
        assert "grid_dependency_wait()" in body, kernel


def test_decode_producers_await_their_last_copies_on_every_way_out():
    """WorkIter::next() is false both at the end of the list and when another role has given up, and a role may give up after a producer
    has issued its last copy: whether the producer itself saw a failure says nothing, so its final wait stands under no condition."""
    text = code("decode.cu")
    producer = text[text.index("warp == 0 || warp >= 16"):text.index("} else if (warp == 1)")]
    loop = producer.index("for (; ok && vw; ++j)")
    depth, i = 0, producer.index("{", loop)
    while True:
        depth += {"{": 1, "}": -1}.get(producer[i], 0)
        i += 1
        if depth == 0:
            break
    after = producer[i:]
    assert "mbar_try_wait" in after and not re.search(r"\bif\b", after)


def test_the_only_build_switches_are_the_give_up_test_builds():
    """No probe that leaves work out, and no path that only other builds reach, is in the sources."""
    found = set()
    for f in SOURCES:
        found |= set(re.findall(r"^[ \t]*#[ \t]*(?:if|ifdef|ifndef|elif)\b[^\n]*?\b(MPFA_\w+)", code(f), flags=re.M))
    assert found == {"MPFA_WAIT_LIMIT_CYCLES", "MPFA_DRAIN_LIMIT_NS", "MPFA_TEST_DROP_V_COPY"}


def test_decode_roles_share_one_waiting_loop():
    """A copy of the loop in each of some thirty waits takes the roles' code past the instruction cache: batches of short contexts were 8 %
    slower for it than with one softmax group fewer in each item."""
    text = code("decode.cu")
    wait = re.search(r"bool wait\(int i, uint32_t parity\) const \{(.*?)\}", text, flags=re.S).group(1)
    assert not re.search(r"\b(for|while)\b", wait) and "wait_longer(" in wait
    assert re.search(r"__noinline__ bool wait_longer\(", text)
    assert text.count("mbar_try_wait_hint(") == 1
