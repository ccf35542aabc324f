"""The digest that ties committed ncu figures to a kernel: it covers the source
and the headers it includes, and nothing that does not reach the compiler."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


def _tree(path, **files):
    for name, text in files.items():
        (path / name.replace("_", ".", 1)).write_text(text)
    return str(path / "k.cu")


def test_digest_follows_headers_and_not_comments(tmp_path):
    import bench
    src = _tree(tmp_path, k_cu='#include <math.h>\n#include "a.cuh"\nint k; // one\n', a_cuh='#include "b.cuh"\nint a;\n',
                b_cuh="/* two\nlines */ int b;\n", c_cuh="int c;\n")
    d = bench.source_digest(src)
    _tree(tmp_path, k_cu='#include <math.h>\n#include "a.cuh"\n\nint k;  // another\n', b_cuh="int b;\n", c_cuh="int d;\n")
    assert bench.source_digest(src) == d  # comments, blanks, a header that is not included
    for name, text in (("a_cuh", '#include "b.cuh"\nint aa;\n'), ("b_cuh", "int bb;\n")):
        _tree(tmp_path, a_cuh='#include "b.cuh"\nint a;\n', b_cuh="int b;\n")
        assert bench.source_digest(src) == d
        _tree(tmp_path, **{name: text})
        assert bench.source_digest(src) != d


def test_digest_of_the_kernels_reaches_their_headers(tmp_path):
    import shutil

    import bench
    csrc = shutil.copytree(os.path.join(ROOT, "paper_1204_4293_gb300", "csrc"), tmp_path / "csrc")
    for kernel, headers in (("fft32.cu", ("fft32_core.cuh", "fft32_tables.cuh", "dft.cuh", "rng.cuh", "tma.cuh", "common.cuh")),
                            ("starlet.cu", ("starlet_math.cuh", "tma.cuh", "common.cuh"))):
        d = bench.source_digest(str(csrc / kernel))
        for h in headers:
            text = (csrc / h).read_text()
            (csrc / h).write_text(text + "\nint changed;\n")
            assert bench.source_digest(str(csrc / kernel)) != d, h
            (csrc / h).write_text(text)
        assert bench.source_digest(str(csrc / kernel)) == d
