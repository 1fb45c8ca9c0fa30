"""A traffic record is tied to all of the code that its kernel was compiled from:
the sources' own headers too."""
import bench


def test_kernel_hash_follows_included_headers(tmp_path, monkeypatch):
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    monkeypatch.setattr(bench, "KERNEL_SOURCES", ("k.cu",))
    src, a, b = tmp_path / "k.cu", tmp_path / "a.cuh", tmp_path / "b.cuh"
    src.write_text('#include <math.h>\n#include "lbm.h"\n#include "a.cuh"\nint f() { return g(); }\n')
    a.write_text('#include "b.cuh"\nint g() { return h(); }\n')
    b.write_text('#include "a.cuh"  // a cycle ends\nint h() { return 1; }\n')
    first = bench.kernel_hash()
    b.write_text('#include "a.cuh"\n// one\nint h() { return 1; }\n')
    assert bench.kernel_hash() == first
    b.write_text('#include "a.cuh"\nint h() { return 2; }\n')
    second = bench.kernel_hash()
    assert second != first
    a.write_text('#include "b.cuh"\nint g() { return h() + 1; }\n')
    assert bench.kernel_hash() not in (first, second)


def test_the_step_kernels_headers_are_covered(tmp_path, monkeypatch):
    import os
    import shutil
    csrc = os.path.join("paper_2311_10827_gb300", "csrc")
    shutil.copytree(os.path.join(bench.ROOT, csrc), tmp_path / csrc)
    want = bench.kernel_hash()
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.kernel_hash() == want
    for name in ("launch.cuh", "d2q9_fp64.cuh", "rcp64.cuh", "lbm_internal.h"):
        path = tmp_path / csrc / name
        text = path.read_text()
        path.write_text(text + "int changed;\n")
        assert bench.kernel_hash() != want, name
        path.write_text(text)
    assert bench.kernel_hash() == want
