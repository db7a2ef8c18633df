"""Which of the two dense kernels a plain pass goes to, on a device of 148 SMs (296 resident CTAs of the single-CTA
kernel, 74 SM pairs): the rule's own arithmetic, compiled for the host."""
import os
import subprocess

import pytest

from paper_2509_24014_b200 import build

# heads of all batch entries, tokens, whether the CTA-pair kernel runs. Where it does not although it is the faster one
# under sustained load, launches with rests between them lose by it.
TABLE = [
    (1, 1024, 0), (256, 4095, 0),                                  # below 4096 tokens
    (1, 4096, 1), (4, 4096, 1), (1, 8192, 1), (1, 16384, 1),       # every cluster split
    (5, 4096, 0), (8, 4096, 0), (4, 5000, 0), (3, 8192, 0), (2, 12288, 0),   # part of a wave, not split
    (10, 4096, 1), (12, 4096, 1), (6, 8192, 1), (3, 16384, 1),     # a wave and split clusters
    (14, 4096, 0), (20, 4096, 0), (28, 4096, 0), (12, 6144, 0),    # short of the power limit
    (32, 4096, 1), (8, 8192, 1), (32, 8192, 1), (256, 4096, 1), (2, 16384, 1), (32, 65536, 1),
    (8, 14000, 0),                                                 # 3.03 waves of clusters, 2.97 of single CTAs
]


# Block-sparse attention, query tiles and whether the kernel whose CTAs have an SM each runs: up to one tile per SM, and
# however short the lists are.
SPARSE_TABLE = [(1, 1), (16, 1), (64, 1), (148, 1), (149, 0), (4096, 0)]


@pytest.fixture(scope="module")
def choice(tmp_path_factory):
    folder = tmp_path_factory.mktemp("dense_choice")
    src, exe = folder / "choice.cpp", folder / "choice"
    src.write_text('#include <cstdio>\n#include <cstdlib>\n#include <cstring>\n#include "dense_choice.h"\n'
                   "using namespace sparsed;\n"
                   "int main(int argc, char** argv) {\n"
                   "  for (int i = 2; i + 2 < argc; i += 3) {\n"
                   "    const long long a = std::atoll(argv[i]), b = std::atoll(argv[i + 1]);\n"
                   "    const int ctas = std::atoi(argv[i + 2]);\n"
                   '    if (std::strcmp(argv[1], "pair") == 0) std::printf("%d\\n", dense_pair_pays(a, static_cast<int>(b), ctas));\n'
                   '    if (std::strcmp(argv[1], "lone") == 0) std::printf("%d\\n", lone_ctas_pay(a, b, ctas));\n'
                   '    if (std::strcmp(argv[1], "sparse") == 0) std::printf("%d\\n", sparse_lone_ctas_pay(a, ctas));\n'
                   "  }\n}\n")
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-I", build.CSRC, str(src), "-o", str(exe)], check=True,
                   capture_output=True, timeout=120)

    def ask(rule, rows):
        args = [rule] + [str(x) for row in rows for x in row]
        return [int(x) for x in subprocess.run([str(exe), *args], check=True, capture_output=True, text=True).stdout.split()]

    return ask


def test_choice(choice):
    got = choice("pair", [(bh, tokens, 296) for bh, tokens, _ in TABLE])
    assert got == [want for _, _, want in TABLE]


def test_sparse_choice(choice):
    assert choice("sparse", [(items, 0, 296) for items, _ in SPARSE_TABLE]) == [want for _, want in SPARSE_TABLE]
    assert choice("sparse", [(items, 0, 0) for items, _ in SPARSE_TABLE]) == [0] * len(SPARSE_TABLE)


def test_no_pairs_without_a_known_device(choice):
    assert choice("pair", [(bh, tokens, ctas) for bh, tokens, _ in TABLE for ctas in (0, 2)]) == [0] * (2 * len(TABLE))
