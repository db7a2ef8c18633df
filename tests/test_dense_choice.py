"""Which kernel an attention call goes to, on a device of 148 SMs (296 resident CTAs of the single-CTA kernel, 74 SM
pairs): the rules' own arithmetic, compiled for the host."""
import os
import subprocess

import pytest

from paper_2509_24014_b200 import build

# The CTA-pair kernel against the single-CTA one: heads of all batch entries, tokens, whether it is the former. Where it
# is not although it is the faster one under sustained load, launches with rests between them lose by it. (Calls of up to
# one query tile per SM are mostly taken by a third kernel first: LONE_TABLE.)
TABLE = [
    (1, 1024, 0), (256, 4095, 0),                                  # below 4096 tokens
    (1, 4096, 1), (4, 4096, 1), (1, 8192, 1), (1, 16384, 1),       # every cluster split
    (5, 4096, 0), (8, 4096, 0), (4, 5000, 0), (3, 8192, 0), (2, 12288, 0),   # part of a wave, not split
    (10, 4096, 1), (12, 4096, 1), (6, 8192, 1), (3, 16384, 1),     # a wave and split clusters
    (14, 4096, 0), (20, 4096, 0), (28, 4096, 0), (12, 6144, 0),    # short of the power limit
    (32, 4096, 1), (8, 8192, 1), (32, 8192, 1), (256, 4096, 1), (2, 16384, 1), (32, 65536, 1),
    (8, 14000, 0),                                                 # 3.03 waves of clusters, 2.97 of single CTAs
]
# The kernel whose CTAs have an SM each, which is asked for first: whether row statistics are recorded, query tiles, keys.
LONE_TABLE = [
    (0, 1, 255, 0), (0, 1, 256, 1), (0, 16, 1024, 1), (0, 98, 256, 1),     # up to two thirds of the SMs
    (0, 99, 256, 0), (0, 148, 1023, 0), (0, 99, 1024, 1), (0, 148, 1024, 1), (0, 128, 8192, 1),
    (0, 149, 256, 0), (0, 149, 8192, 0), (0, 480, 1900, 0),                # more tiles than SMs
    (1, 148, 255, 0), (1, 99, 256, 1), (1, 148, 256, 1), (1, 149, 8192, 0),
]
# The dense choice as a whole: whether row statistics are recorded, heads, tokens, kernel.
SINGLE, PAIR, LONE = range(3)
DENSE_TABLE = [
    (0, 2, 255, SINGLE), (0, 2, 256, LONE), (0, 2, 1024, LONE), (0, 37, 512, SINGLE), (0, 18, 1024, LONE),
    (0, 32, 1900, SINGLE), (0, 1, 4096, LONE), (0, 4, 4096, LONE), (0, 5, 4096, SINGLE), (0, 1, 16384, LONE),
    (0, 10, 4096, PAIR), (0, 32, 8192, PAIR), (0, 8, 14000, SINGLE),
    (1, 37, 192, PAIR), (1, 2, 1024, LONE), (1, 37, 512, LONE), (1, 38, 512, PAIR), (1, 16, 2944, PAIR), (1, 32, 4096, PAIR),
]
# Block-sparse attention on the kernel whose CTAs have an SM each: query tiles, average list in blocks (None: not known), block size.
SPARSE_TABLE = [
    (1, None, 128, 1), (74, None, 128, 1), (74, 0.1, 32, 1), (74, 1, 64, 1),   # up to half of the SMs: any lists
    (75, None, 128, 0), (75, 3.9, 128, 0), (75, 4, 128, 1), (98, 4, 128, 1), (98, None, 64, 1), (98, 0.1, 32, 1),
    (99, 4, 128, 0), (99, 15.9, 128, 0), (99, 16, 128, 1), (148, 16, 128, 1),  # beyond two thirds
    (99, None, 64, 0), (148, 7.9, 64, 0), (148, 8, 64, 1), (148, 15.9, 32, 0), (148, 16, 32, 1),
    (149, 64, 128, 0), (149, 64, 32, 0), (149, None, 64, 0),
]


@pytest.fixture(scope="module")
def choice(tmp_path_factory):
    folder = tmp_path_factory.mktemp("dense_choice")
    src, exe = folder / "choice.cpp", folder / "choice"
    src.write_text('#include <cstdio>\n#include <cstdlib>\n#include <cstring>\n#include "dense_choice.h"\n'
                   "using namespace sparsed;\n"
                   "int main(int argc, char** argv) {\n"
                   "  auto arg = [&](int i) { return std::atoll(argv[i]); };\n"
                   "  auto is = [&](const char* rule) { return std::strcmp(argv[1], rule) == 0; };\n"
                   "  const int n = is(\"pair\") ? 3 : is(\"lone\") || is(\"dense\") ? 4 : 6;\n"
                   "  for (int i = 2; i + n <= argc; i += n)\n"
                   '    std::printf("%d\\n", is("pair")   ? dense_pair_pays(arg(i), arg(i + 1), arg(i + 2))\n'
                   '                        : is("lone") ? lone_ctas_pay(arg(i), arg(i + 1), arg(i + 2), arg(i + 3))\n'
                   '                        : is("dense") ? static_cast<int>(choose_dense_kernel(arg(i), arg(i + 1), arg(i + 2), arg(i + 3)))\n'
                   "                                     : sparse_lone_ctas_pay(arg(i), arg(i + 1), arg(i + 2), arg(i + 3),\n"
                   "                                                            arg(i + 4), arg(i + 5)));\n}\n")
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-I", build.CSRC, str(src), "-o", str(exe)], check=True,
                   capture_output=True, timeout=120)

    def ask(rule, rows):
        args = [rule] + [str(x) for row in rows for x in row]
        return [int(x) for x in subprocess.run([str(exe), *args], check=True, capture_output=True, text=True).stdout.split()]

    return ask


def test_choice(choice):
    got = choice("pair", [(bh, tokens, 296) for bh, tokens, _ in TABLE])
    assert got == [want for _, _, want in TABLE]


def test_lone_choice(choice):
    assert choice("lone", [(*row[:3], 296) for row in LONE_TABLE]) == [row[3] for row in LONE_TABLE]
    assert choice("lone", [(*row[:3], 0) for row in LONE_TABLE]) == [0] * len(LONE_TABLE)


def test_dense_choice(choice):
    assert choice("dense", [(*row[:3], 296) for row in DENSE_TABLE]) == [row[3] for row in DENSE_TABLE]
    assert choice("dense", [(*row[:3], 0) for row in DENSE_TABLE]) == [PAIR if row[0] else SINGLE for row in DENSE_TABLE]


def test_sparse_choice(choice):
    def ask(ctas):
        rows = [(items, items * 128 // bs) for items, _, bs, _ in SPARSE_TABLE]   # one head: a list per query block
        return choice("sparse", [(items, 0 if blocks is None else int(n * blocks + 0.5), n, n, bs, ctas)
                                 for (items, n), (_, blocks, bs, _) in zip(rows, SPARSE_TABLE)])

    assert ask(296) == [row[3] for row in SPARSE_TABLE]
    assert ask(0) == [0] * len(SPARSE_TABLE)
    # counts that cannot be: more entries than the rows have blocks (a buffer's room), a field nobody set
    assert choice("sparse", [(148, 1 << 40, 148, 148, 128, 296), (148, 1 << 62, 148, 15, 128, 296),
                             (148, -1, 148, 148, 128, 296), (148, -(1 << 63), 592, 592, 32, 296)]) == [1, 0, 0, 0]


def test_no_pairs_without_a_known_device(choice):
    assert choice("pair", [(bh, tokens, ctas) for bh, tokens, _ in TABLE for ctas in (0, 2)]) == [0] * (2 * len(TABLE))
