"""The ncu figures that bench.py reports belong to every file that the captured kernels are compiled from."""
import os
import re

import bench

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = "paper_1910_02858_gb300/csrc/"


def test_hash_covers_all_included_sources():
    todo, seen = [CSRC + f for f in ("k_dg_f64.cu", "k_dg_f32.cu", "k_adj_f64.cu")], set()
    while todo:
        f = todo.pop()
        if f in seen or not os.path.exists(os.path.join(ROOT, f)):
            continue
        seen.add(f)
        text = open(os.path.join(ROOT, f), encoding="utf-8").read()
        todo += [CSRC + m for m in re.findall(r'#include "([^"]+)"', text)]
    headers = {f for f in seen if not f.endswith(".cu")}
    assert len(headers) >= 10 and headers <= set(bench.KERNEL_SOURCES), headers - set(bench.KERNEL_SOURCES)


def test_affine_elements_move_fewer_words():
    # the headline mesh: 36 + 117 f words per DOF and stage, f = 3 / 8
    assert bench.algorithmic_per_dof(8, 8)[0] - bench.AFFINE_WORDS * 8 == 8 * (36 + 117 * 3 / 8)
