"""Rules of the SELL layouts that need no GPU, compiled for the host from the library's own header."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"


def run(tmp_path, body):
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text('#include "common.cuh"\n#include <cstdint>\n#include <cstdio>\nusing namespace cpc;\n'
                   "#define OK(c) if (!(c)) { std::printf(\"%%d: %%s\\n\", __LINE__, #c); return 1; }\n"
                   "int main() {\n%s\nreturn 0;\n}\n" % body)
    subprocess.run([NVCC, "-std=c++17", "-O1", "--expt-relaxed-constexpr", "-I", os.path.join(ROOT, "paper_1205_6113_gb300", "csrc"), str(src),
                    "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


@pytest.mark.skipif(not os.path.exists(NVCC), reason="no nvcc")
def test_columns_and_their_marks_take_every_int32(tmp_path):
    """A column up to the last of the largest matrix is taken as it is; marked, it is skipped from a zero
    guess and found again; padding is neither."""
    run(tmp_path, """
    for (int64_t j : {0ll, 1ll, (1ll << 30) - 1, 1ll << 30, (1ll << 30) + 1, (1ll << 31) - 2}) {
        const int c = (int)j, m = mark_later(c);
        OK(takes(c) && !is_later(c) && marked_col(c) == c && c != -1)
        OK(!takes(m) && is_later(m) && marked_col(m) == c && m != -1)
    }
    OK(!takes(-1) && !is_later(-1))
""")


def test_shared_arrays_of_vector_loads_are_aligned():
    """ldv reads up to 16 bytes at a time: every shared array that it reads is declared so."""
    import re
    text = open(os.path.join(ROOT, "paper_1205_6113_gb300", "csrc", "batched.cu")).read()
    shared = dict((name, decl) for decl, name in re.findall(r"((?:extern )?__shared__ [^;\n]*?\b(\w+)\[)", text))
    alias = dict(re.findall(r"double\* (\w+) = (ksm)\b", text))
    read = {alias.get(a, a) for a in re.findall(r"\bldv<\w+>\((\w+)", text)} & set(shared)
    assert read == {"fs", "ksm"}
    decls = [d for d in re.findall(r"(?:extern )?__shared__ [^;\n]*", text) if re.search(r"\b(fs|ksm)\[", d)]
    assert len(decls) == 5 and all("__align__(16)" in d for d in decls), decls


@pytest.mark.skipif(not os.path.exists(NVCC), reason="no nvcc")
def test_layouts_stay_within_their_offsets(tmp_path):
    """Two paddings per chunk can carry a layout past 32-bit offsets where one did not; the count that decides
    is taken in 64 bits (67,108,864 chunks of 32 entries are one entry too many)."""
    run(tmp_path, """
    OK(sell_fits(0) && sell_fits(INT32_MAX) && !sell_fits((int64_t)INT32_MAX + 1))
    OK(!sell_fits((int64_t)67108864 * 32) && sell_fits((int64_t)67108863 * 32))
""")


@pytest.mark.skipif(not os.path.exists(NVCC), reason="no nvcc")
def test_sides_of_entries_are_told_apart(tmp_path):
    """The layout checker's rules on sound and planted entries: the part of earlier groups, the mark of later
    ones, a column that is not the entry's, an entry dropped as padding."""
    run(tmp_path, """
    for (int gr = 0; gr < 3; ++gr)
        for (int gc = 0; gc < 3; ++gc) {
            if (gc == gr) continue;
            OK(part_holds(gc < gr, gr, gc) && !part_holds(gc > gr, gr, gc))
            for (int c : {0, 7, 1 << 30}) {
                const int right = gc > gr ? mark_later(c) : c, wrong = gc > gr ? c : mark_later(c);
                OK(mark_holds(right, c, gr, gc) && !mark_holds(wrong, c, gr, gc))
                OK(!mark_holds(-1, c, gr, gc) && !mark_holds(right, c + 1, gr, gc))
            }
        }
""")
