"""The rules that keep overlapping launches apart (csrc/launch.cuh), checked on the source: what they prevent is a block that waits
for good, so nothing here runs a kernel."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2409_09083_b200", "csrc")


def sources():
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cuh", ".cu")):
            with open(os.path.join(CSRC, f)) as h:
                yield f, re.sub(r"//[^\n]*", "", h.read())


def body(text, at):
    """The braces' content that follows position `at`."""
    begin = text.index("{", at)
    depth = 0
    for i in range(begin, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[begin:i + 1]
    raise AssertionError("unbalanced braces")


def functions(pattern):
    """{name: body} of the functions whose head matches (the last name in front of the parameter list is the function's)."""
    out = {}
    for f, text in sources():
        for m in re.finditer(pattern, text):
            out[m.group("name")] = body(text, text.index(")", m.end()))
    return out


KERNELS = functions(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s+)?(?P<name>\w+)\(")
SETUP = functions(r"__device__ __forceinline__ void (?P<name>setup)\(")["setup"]
LAUNCHED = {n for _, t in sources() for n in re.findall(r"(?<!\w)launch\(\s*(?:sp::)?(\w+)", t)} & set(KERNELS) | \
           {"conv_split_kernel"}                             # launched through a table of its instances


def inlined(name):
    return re.sub(r"(?<!\w)setup\([^;]*;", lambda m: SETUP, KERNELS[name])


def test_kernels_were_found():
    assert {"fwd_group_tc_kernel", "bwd_group_tc_kernel", "conv_tc_rows_kernel", "filter_grad_tc_rows_kernel", "conv_split_kernel",
            "fgrad_split_kernel", "conv_rows_kernel", "reduce_sgd_tc_kernel"} <= LAUNCHED
    assert "tmem_alloc" in SETUP and "__syncthreads" in SETUP.split("tmem_alloc")[1]


@pytest.mark.parametrize("name", sorted(KERNELS))
def test_the_next_launch_is_let_in_behind_the_allocation_of_tensor_memory(name):
    text = inlined(name)
    if "tmem_alloc" in text and "next_launch()" in text:
        assert text.index("next_launch()") > text.index("__syncthreads", text.index("tmem_alloc")), name


@pytest.mark.parametrize("name", sorted(LAUNCHED))
def test_launches_that_may_overlap_wait_for_the_previous_ones(name):
    """(Before anything but their own set-up in shared and tensor memory: reads of global memory go through __ldg, `A.` pointers or
    asynchronous copies, none of which stands in front of the wait.)"""
    text = inlined(name)
    assert "previous_launches()" in text, name
    front = text[:text.index("previous_launches()")]
    assert not re.search(r"__ldg|tma_load|bulk_g2s|cp_async|atomic|A\.\w+\[", front), name


def asm_statements():
    """(file, instructions, outputs) of every asm statement: the instructions of its template, comments and declarations left out."""
    for f, text in sources():
        for m in re.finditer(r"\basm\s*(?:volatile)?\s*\(", text):
            depth, i = 1, m.end()
            while depth:
                i += 1
                depth += {"(": 1, ")": -1}.get(text[i], 0)
            # (operands behind the first colon that stands outside the strings)
            parts = re.split(r":(?=(?:[^\"]*\"[^\"]*\")*[^\"]*$)", text[m.end():i])
            template = "".join(re.findall(r'"((?:[^"\\]|\\.)*)"', parts[0]))
            code = [c.strip(" {}\t") for c in re.split(r";|\\n|\\t", template)]
            yield f, [c for c in code if c and not c.startswith(".reg")], parts[1] if len(parts) > 1 else ""


def test_outputs_written_before_the_last_input_is_read_have_registers_of_their_own():
    """The compiler may give an output the register of an input unless the output is marked "=&r" (or "+r"): in a statement of several
    instructions an output of any but the last one has to be, as a later instruction may still read the input."""
    seen = 0
    for f, code, outputs in asm_statements():
        names = re.findall(r'"([=+]&?\w)"\s*\(', outputs)
        last = max((i for i, c in enumerate(code) if "%" in c), default=0)
        for i, c in enumerate(code[:last]):
            written = {int(n) for n in re.findall(r"%(\d+)", c)} & set(range(len(names)))
            seen += len(written)
            assert all("&" in names[n] or "+" in names[n] for n in written), (f, c, [names[n] for n in written])
    assert seen >= 16
