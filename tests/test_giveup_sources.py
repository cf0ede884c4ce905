"""What a kernel does after a bounded wait has given up, read from its source (no GPU: no test makes a real kernel
lose a signal)."""
import os
import re

import pytest

import paper_2310_01655_b200 as psk

CSRC = os.path.join(os.path.dirname(psk.__file__), "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def loops(text):
    """(header, body) of every for loop with a braced body."""
    for m in re.finditer(r"\bfor \(([^{}]*?)\) \{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(1), text[m.end():i]


@pytest.mark.parametrize("name", ["psk_tc.cu", "psk_tc_bwd.cu", "psk_tc_state.cu", "psk_lt_tc.cu", "psk_sketch8_tc.cu"])
def test_a_later_wait_does_not_hide_one_that_gave_up(name):
    """In a loop that runs on after a wait gave up, `ok` keeps that: it is only ever and-ed."""
    for header, body in loops(source(name)):
        if re.search(r"&& ok\b", header):            # (such a loop ends instead)
            continue
        for stmt in re.findall(r"\bok = mbar_(?:wait|spin)\([^;]*;", body):
            inner = next((h for h, b in loops(body) if stmt in b and re.search(r"&& ok\b", h)), None)
            follows = body[body.index(stmt) + len(stmt):].lstrip()
            assert inner or "&& ok;" in stmt or follows.startswith("if (!ok) break;"), (header, stmt)


@pytest.mark.parametrize("name,calls", [
    ("psk_tc_bwd.cu", [r"refill\(C\);", r"load_m\(tp \+ 1,", r"load_y\(tp \+ 1\);", r"mbar_expect_tx\(&bar_again,"]),
    ("psk_tc.cu", [r"mbar_expect_tx\(&bar_q, 16384\);", r"mbar_expect_tx\(&bar_feat\[kZStages", r"load_k\(P, P\);", r"load_v\(P, P\);",
                   r"load_k\(nx,", r"mbar_expect_tx\(&bar_feat\[buf\]", r"mbar_arrive\(&bar_feat\[buf\]\);"]),
    ("psk_tc_state.cu", [r"load_x\(j \+ 2\);", r"load_y\(j \+ 1\);", r"tma_store_4d\(&mapH,"]),
    ("psk_sketch8_tc.cu", [r"load_x\(tile \+", r"load_d\(tile \+", r"tma_store_tile\(&map"]),
])
def test_no_copy_is_asked_for_after_a_wait_gave_up(name, calls):
    """Every copy that is asked for behind a wait has `ok` in the condition in front of it.  (Its barrier's phase may still be
    open: one more arrival with bytes outstanding, and a second copy into the buffer.)"""
    text = source(name)
    for call in calls:
        found = [m.start() for m in re.finditer(call, text)]
        assert found, call
        for at in found:
            # the nearest `if (...)` before the call
            conditions = re.findall(r"\bif (?:constexpr )?\((.*)\)", text[:at][-400:])
            conditions = [c for c in conditions if "L::" not in c or "ok" in c]
            assert conditions and re.search(r"\bok\b", conditions[-1]), (name, call, conditions[-1:])


@pytest.mark.parametrize("name", ["psk_tc.cu", "psk_tc_bwd.cu", "psk_tc_state.cu", "psk_lt_tc.cu", "psk_sketch8_tc.cu"])
def test_tensor_memory_is_read_by_whole_warps(name):
    """Loads and stores of tensor memory need every lane of a warp; after a wait gave up in some lanes only, `ok` differs."""
    text = source(name)
    for m in re.finditer(r"\bif \((?:[^{};]*\W)?ok\b[^{};]*\) \{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        assert not re.search(r"\btmem_(?:ld|st)", text[m.end():i]), (name, m.group(0))


def test_the_networks_feeders_stop_asking_for_copies():
    """The learnable sketch's issuing lanes leave their loop where a wait in front of a copy gave up."""
    text = source("psk_learned_tc.cu")
    for wait, copy, leave in ((r"bar_t, k & 1", r"load\(i \+ 2\);", "break;"), (r"bar_free, \(k - 1\) & 1", r"load\(i \+ 1\);", "break;"),
                              (r"bar_rd\[1\], \(k - 1\) & 1", r"load_lo\(i\);", "return false;")):
        assert re.search(r"!mbar_spin\(&" + wait + r", status, kErrMma\)+ " + leave + r".{0,200}?" + copy, text, re.S), copy


def test_tensor_memory_is_given_back_after_the_teardown():
    """Every kernel that issues MMAs goes through cta_teardown() between its last block-wide barrier and the release of its
    tensor memory: MMAs and copies of a CTA that gave up a wait must not outlive it."""
    kernels = 0
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith(".cu"):
            continue
        text = source(name)
        for m in re.finditer(r"\btmem_dealloc\(", text):
            kernels += 1
            before = text[:m.start()]
            assert before.rfind("cta_teardown") > before.rfind("__syncthreads"), name
    assert kernels >= 10
