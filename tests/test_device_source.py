"""Orderings that a run cannot show to be there: checked in the text of the kernels."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_07609_b200", "csrc")


def _text(name):
    return open(os.path.join(CSRC, name)).read()


def _body(text, name):
    start = re.search(r"\b%s\([^;{]*\{" % name, text).end()
    depth, i = 1, start
    while depth:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        i += 1
    return text[start:i]


def test_a_token_operand_made_by_a_pair_is_handed_over_at_cluster_scope():
    """CTA 1 writes its half with ordinary stores, CTA 0 issues the MMAs that read it: a release and an acquire whose scope
    holds both CTAs have to lie between (an arrival without a scope releases to its own CTA only)."""
    dec, tc = _text("gemm_dec.cuh"), _text("gemm_tc.cuh")
    arrive = re.search(r"if constexpr \(PAIR\) (\w+)\(&g_dec\.b_made\)", dec).group(1)
    wait = re.search(r"PAIR \? (\w+)\(c, &g_dec\.b_made", dec)
    assert wait, "pairs wait for the made operand with a wait of their own"
    out, back = _body(tc, arrive), _body(tc, wait.group(1))
    assert re.search(r"arrive\.release\.cluster|fence\.(release\.sync_restrict::shared::cta|acq_rel)\.cluster.*arrive\.relaxed\.cluster", out, re.S), arrive
    assert re.search(r"try_wait\.parity\.acquire\.cluster|try_wait\.parity\.relaxed\.cluster.*fence\.(acquire\.sync_restrict::shared::cluster|acq_rel)\.cluster",
                     back, re.S), wait.group(1)


def test_the_control_cta_leaves_by_one_threads_clock():
    """Threads that each compare their own clock leave the idle loop in different turns, and the CTA's barriers no longer match."""
    body = _body(_text("control.cuh"), "control_phase")
    by_thread_0 = "".join(re.findall(r"if \(tid == 0\) \{.*?\n    \}", body, re.S))
    assert body.count("- idle_t0") == by_thread_0.count("- idle_t0") == 1


def test_scheduler_and_phases_go_by_one_row_limit_for_small_steps():
    """The scheduler decides who applies RoPE, the phases who clears its input: two limits would drop one or the other."""
    control, dec = _text("control.cuh"), _text("gemm_dec.cuh")
    assert re.search(r"const int fuse = c\.dec_small && T <= DEC_SMALL_ROWS\b", control)
    assert re.search(r"bool dec_small\(.*\{ return c\.dec_small && T <= DEC_SMALL_ROWS; \}", dec)


def test_registers_of_a_tensor_memory_load_are_not_touched_before_the_wait():
    """They hold nothing until tcgen05.wait::ld.  So the wait is part of the load's statement, or it names the registers (+r) and stands
    behind the load in the same block: no branch, no way around a loop and no change of type between the two, each of which
    may be a copy."""
    texts = {f: re.sub(r"//[^\n]*", "", _text(f)) for f in sorted(os.listdir(CSRC)) if f.endswith((".cuh", ".cu"))}
    wrappers, n_loads = [], 0
    for text in texts.values():
        for st in re.finditer(r"asm volatile\((.*?)\);", text, re.S):
            code = st.group(1)
            if "tcgen05.ld." in code:
                n_loads += 1
                if "tcgen05.wait::ld" in code:
                    assert code.index("tcgen05.ld.") < code.index("tcgen05.wait::ld")
                    continue
                name, args = re.findall(r"void (\w+)\(([^{;]*)\) \{\s", text[:st.start()])[-1]
                assert re.search(r"uint32_t \(&\w+\)\[\d+\]", args), f"{name}: destinations of another type than the instruction's"
                wrappers.append(name)
            elif "tcgen05.wait::ld" in code:
                assert "+r" in code or "BLINK_RW" in code, "a wait that names no registers orders nothing that uses them"
    assert n_loads >= 2
    for name in wrappers:
        for f, text in texts.items():
            for call in re.finditer(r"\b%s\(([^;{]*), (\w+)\);" % name, text):
                depth, i = 0, call.end()
                while depth >= 0:   # to the end of the block that the load stands in
                    depth += {"{": 1, "}": -1}.get(text[i], 0)
                    i += 1
                head = text[:call.start()].rstrip()
                assert head[-1] in ";{}", f"{f}: {call.group(0)} under a condition"
                assert re.search(r"tmem_wait_ld\w*\([^;]*\b%s\b[^;]*\);" % call.group(2), text[call.end():i]), f"{f}: {call.group(0)} is not waited for in its block"
