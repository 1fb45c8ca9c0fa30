"""The adjoint recorder's buffers are one block of device memory where one that
large can be had, and separate blocks where only those fit (a fragmented or
nearly full device), with a host stand-in for the allocator."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2311_10827_gb300", "csrc")
DRIVER = r"""
#include "parts.h"
#include <stdio.h>
#include <stdlib.h>
// argv: largest block, total budget, part sizes; prints what is held and how
int main(int argc, char **argv)
{
    const long largest = atol(argv[1]);
    long left = atol(argv[2]), live = 0;
    const int n = argc - 3;
    void *p[16] = {}, *blocks[16];
    wblbm::Part part[16];
    for (int k = 0; k < n; ++k) part[k] = {&p[k], (size_t)atol(argv[3 + k])};
    int calls = 0;
    auto alloc = [&](void **q, size_t b) {
        ++calls;
        if ((long)b > largest || (long)b > left) return false;
        if (posix_memalign(q, 256, b)) return false;
        left -= (long)b;
        ++live;
        return true;
    };
    auto release = [&](void *q) { free(q); --live; };
    const bool ok = wblbm::alloc_parts(part, n, blocks, alloc, release);
    int held = 0, apart = 1;
    for (int k = 0; k < n; ++k) {
        held += blocks[k] != nullptr;
        if (!ok) continue;
        if ((size_t)p[k] % 256) apart = 0;
        for (int j = 0; j < k; ++j)  // no two parts overlap
            if ((char *)p[j] < (char *)p[k] + part[k].bytes &&
                (char *)p[k] < (char *)p[j] + part[j].bytes)
                apart = 0;
        for (size_t b = 0; b < part[k].bytes; ++b) ((char *)p[k])[b] = (char)k;
    }
    printf("%d %d %ld %d %d\n", ok, held, live, apart, calls);
    for (int k = 0; k < n; ++k) free(blocks[k]);
    return 0;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    d = tmp_path_factory.mktemp("parts")
    src, exe = str(d / "parts.cc"), str(d / "parts")
    with open(src, "w") as fh:
        fh.write(DRIVER)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-fsanitize=address", "-I", CSRC, src,
                    "-o", exe], check=True)

    def call(largest, budget, *sizes):
        out = subprocess.run([exe, str(largest), str(budget), *map(str, sizes)], check=True,
                             capture_output=True, text=True).stdout.split()
        return dict(zip(("ok", "held", "live", "apart", "calls"), map(int, out)))
    return call


def test_one_block_where_it_fits(run):
    assert run(10 ** 6, 10 ** 6, 1000, 24, 256, 7) == dict(ok=1, held=1, live=1, apart=1, calls=1)


def test_separate_blocks_where_one_does_not(run):
    r = run(2000, 10 ** 6, 1000, 2000, 24)  # 3328 together
    assert r == dict(ok=1, held=3, live=3, apart=1, calls=4)


def test_nothing_is_held_when_a_part_does_not_fit(run):
    r = run(2000, 10 ** 6, 1000, 24, 2001, 8)
    assert r["ok"] == 0 and r["held"] == 0 and r["live"] == 0


def test_the_recorder_uses_it():
    with open(os.path.join(CSRC, "lbm_capi.cu")) as fh:
        text = fh.read()
    body = text[text.index("int lbm_adjoint_create("):text.index("int lbm_adjoint_forward(")]
    assert "alloc_parts(" in body and "cudaMalloc(" in body and body.count("cudaMalloc(") == 1
