"""Kernels launched before the grid in front of them has ended (launch_pdl) read its
results through the read-only path, and the compiler may place such loads
anywhere their address is known.  So every one of these kernels takes the index
along x of its block or of its thread from the wait itself, uses no other, and
reads nothing before it; a pointer that is read without that index goes through
after_wait."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2311_10827_gb300", "csrc")


def sources():
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh")):
            with open(os.path.join(CSRC, f)) as fh:
                yield f, re.sub(r"//[^\n]*", "", fh.read())


def kernels(text):
    """(name, parameters, body) of the __global__ functions."""
    for m in re.finditer(r"__global__[^{;]*?(\w+)\(const (?:StepParams|BatchCase)", text):
        i = text.index("(", m.end(1))
        j = text.index("{", i)
        depth, k = 1, j + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[k], 0)
            k += 1
        yield m.group(1), text[i:j], text[j:k]


def test_every_kernel_of_launch_pdl_takes_an_index_from_the_wait():
    launched, waiting = set(), {}
    for f, text in sources():
        launched |= set(re.findall(r"launch_pdl\((\w+)", text)) - {"void"}
        for name, params, body in kernels(text):
            if "pdl_wait(" in body:
                waiting[name] = (f, params, body)
    assert launched and launched == set(waiting)
    for name, (f, params, body) in waiting.items():
        where = f"{f}: {name}"
        assert body.count("pdl_wait(") == 1, where
        index = re.search(r"pdl_wait\((blockIdx\.x|threadIdx\.x)\)", body).group(1)
        assert body.count(index) == 1, where
        before = body[:body.index("pdl_wait(")]
        # only shared-memory declarations and constants stand before it
        rest = re.sub(r"(__shared__|constexpr|using)[^;]*;", "", before)
        assert re.fullmatch(r"\{\s*(const (int|unsigned) \w+ =)?\s*", rest), (where, rest)


def test_uniform_reads_come_after_the_wait():
    """What is read without a block index: the offset storage's scales."""
    n = 0
    for f, text in sources():
        for name, params, body in kernels(text):
            if "pdl_wait(" not in body:
                continue
            for arg in re.findall(r"__ldg\((\w[\w.]*)(?: \+ \d)?\)", body):
                assert f"{arg} = after_wait(" in body, (f, name, arg)
                n += 1
            assert not re.search(r"\*\s*target|target\[|src\.sc\[", body), (f, name)
            assert "src.sc" not in body.replace("after_wait(src.sc)", ""), (f, name)
            n += body.count("after_wait(src.sc)")
    assert n >= 11


def test_the_wait_defines_the_index():
    with open(os.path.join(CSRC, "launch.cuh")) as fh:
        text = fh.read()
    assert re.search(r'asm volatile\("griddepcontrol\.wait;" : "\+r"\(index\)\s*::\s*"memory"\)', text)
    assert re.search(r'asm volatile\("" : "\+l"\(p\)\)', text)


def test_the_tiles_take_the_threads_index_from_their_kernel():
    """A kernel that passes its thread index on: the march has no other."""
    for f, text in sources():
        for m in re.finditer(r"void (d2q9_tile\w*)\(([^)]*)\)\s*\{", text):
            assert re.search(r"\btx$", m.group(2)), m.group(1)
            k, depth = m.end(), 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[k], 0)
                k += 1
            assert "threadIdx.x" not in text[m.end():k], m.group(1)
