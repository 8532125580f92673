"""Statements whose order or operand marks the results rest on and that no run
is sure to show, read from the kernels' source."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2206_05761_gb300", "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def body_of(src, head):
    """The braces' block that follows `head`."""
    i = src.index("{", src.index(head))
    depth = 0
    for k in range(i, len(src)):
        depth += {"{": 1, "}": -1}.get(src[k], 0)
        if depth == 0:
            return src[i:k + 1]
    raise AssertionError(head)


def test_the_encode_orders_its_thresholds_before_they_are_read():
    b = body_of(source("kernels.cuh"), "void encode_tile(")
    write = b.index("sthr[w][j][q] = ")
    read = b.index("sthr[w][0]", write)
    between = b[write:read]
    assert "__syncwarp(" in between or "__syncthreads(" in between


def asm_statements(src):
    """(text, outputs, inputs) of every asm statement: operands as constraint
    strings in order."""
    out = []
    for m in re.finditer(r"\basm\b(?:\s+volatile)?\s*\(", src):
        k, depth, quote = m.end(), 1, False
        while depth:
            c = src[k]
            if c == '"':
                quote = not quote
            elif not quote:
                depth += {"(": 1, ")": -1}.get(c, 0)
            k += 1
        stmt = src[m.end():k - 1]
        # outside of strings, colons separate text, outputs, inputs, clobbers
        parts, cur, quote = [], "", False
        for c in stmt:
            if c == '"':
                quote = not quote
            if c == ":" and not quote:
                parts.append(cur)
                cur = ""
            else:
                cur += c
        parts.append(cur)
        strings = [re.findall(r'"([^"]*)"', x) for x in parts]
        strings += [[]] * (3 - len(strings))
        out.append(("".join(strings[0]), strings[1], strings[2]))
    return out


def test_outputs_written_before_an_input_is_read_share_no_register():
    checked = 0
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cuh", ".cu", ".h")):
            continue
        for text, outs, ins in asm_statements(source(name)):
            stmts = [re.sub(r"\.reg[^;]*", "", t) for t in text.replace("\\n", "").replace("\\t", "").split(";")]
            uses = [[int(x) for x in re.findall(r"%(\d+)", t)] for t in stmts]
            inputs = range(len(outs), len(outs) + len(ins))
            for o, mark in enumerate(outs):
                first = [i for i, u in enumerate(uses) if o in u]
                later = [x for u in uses[first[0] + 1:] for x in u if x in inputs]
                checked += 1
                if later:
                    assert "&" in mark, (name, text, o, mark)
    assert checked > 10


def test_the_reader_of_asm_statements_sees_the_fault():
    bad = 'asm("add.cc.u32 %0, %2, 0; addc.u32 %1, %3, 0;" : "=r"(a), "=r"(b) : "r"(c), "r"(d));'
    (text, outs, ins), = asm_statements(bad)
    assert outs == ["=r", "=r"] and ins == ["r", "r"] and text.count(";") == 2


def test_no_load_can_move_above_the_wait_for_the_kernel_ahead():
    # an asm statement that loads is volatile, as the wait is: the compiler
    # keeps volatile statements in order
    loads = 0
    for name in ("common.cuh", "kernels.cuh", "skip.cuh"):
        for m in re.finditer(r"\basm\b\s*(volatile)?\s*\(\s*\"(?:ld\.|\{?\s*ld\.)", source(name)):
            loads += 1
            assert m.group(1), (name, source(name)[m.start():m.start() + 80])
    assert loads >= 4
    # a launch whose kernel gets no state to read first is an ordinary one: the
    # bed's encode and flags while the handle is made, the flags on demand
    src = source("engine.cuh")
    assert re.search(r"bool pdl_ = false;", src)
    init = body_of(src, "hwfv1_status init(")
    assert init.index("pdl_ = ") > max(init.index("encode_passes("), init.index("lk(k_flag"))
    assert "lk(" not in init[init.index("pdl_ = "):]
    assert "lk(" not in body_of(src, "void ensure_sig_words(")


def test_a_dry_pass_starts_with_an_empty_queue():
    # every host function that launches the dry pass or a step outside a graph
    # empties the queue first: by a new end time (advance, uniform steps) or on
    # its own; appended to an earlier queue, the leaves would leave the list
    src = source("engine.cuh")
    for head, start in (("hwfv1_status step()", "launch_fv1("), ("hwfv1_status profile_step(", "launch_step("),
                        ("hwfv1_status profile_update(", "launch_encode("),
                        ("hwfv1_status advance(", "launch_step("),
                        ("hwfv1_status advance_uniform(", "launch_step_uniform(")):
        b = body_of(src, head)
        first = min(b.find(x) for x in ("new_queue(", "k_set_tend<<<") if x in b)
        assert -1 < first < b.index(start), head


def test_uniform_steps_leave_no_length_to_the_adaptive_list():
    # the uniform steps' M counts a list of their own; hwfv1_step reads M entries
    # of the adaptive list, of which a handle without a traversal has none
    b = body_of(source("engine.cuh"), "hwfv1_status advance_uniform(")
    assert re.search(r"cudaMemsetAsync\(&st_->M, 0, sizeof\(uint32_t\)", b[b.rindex("launch_step_uniform("):])
