"""The bench's work models of the FP64 form's kernels: each is scored at its own
operations and rate, and the tree's compositions are split between the leaf
kernel and the tree where both run."""
import os
import re
import sys

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402

ITERS, N_H = np.array([5, 6, 4]), np.array([64, 128, 250])
INTERVALS = float(np.sum(ITERS * N_H))


def _rates(kt):
    _, k = bench.roofline(dict(kt, k_outputs=(0.1, 1)), ITERS, N_H, 1457, 0,
                          peaks={"fp32_tflops": 70.0, "fp64_tflops": 1.0})
    return k


def test_kernels_are_scored_at_the_fp64_rate():
    ms = {"k_condense_fp64": 21.0, "k_tree_fp64": 8.0, "k_recover_fp64": 1.8, "k_point_fp64": 4.0}
    k = _rates({name: (t, 6) for name, t in ms.items()})
    points = float(np.sum(ITERS * (3 * N_H + 1)))
    work = {"k_condense_fp64": bench.flops_condense_fp64_interval() * INTERVALS,
            "k_tree_fp64": (bench.flops_compose() + bench.flops_tree_down()) * INTERVALS,
            "k_recover_fp64": bench.flops_recover_fp64_interval() * INTERVALS,
            "k_point_fp64": bench.flops_point_fp64() * points}
    for name, w in work.items():
        assert k[name]["bound"] == "alu" and k[name]["peak"] == 1.0, name
        assert abs(k[name]["achieved"] - w / (ms[name] * 1e-3) / 1e12) <= 1e-9 * k[name]["achieved"], name


def test_compositions_are_split_with_the_leaf_kernel():
    k = _rates({"k_tree_leaf_fp64": (5.0, 6), "k_tree_fp64": (3.0, 6)})
    leaf = float(np.sum(ITERS * (N_H - np.ceil(N_H / 16))))   # one composition less than intervals in a block
    assert abs(k["k_tree_leaf_fp64"]["achieved"] - bench.flops_compose() * leaf / 5e-3 / 1e12) <= 1e-9
    rest = bench.flops_compose() * (INTERVALS - leaf) + bench.flops_tree_down() * INTERVALS
    assert abs(k["k_tree_fp64"]["achieved"] - rest / 3e-3 / 1e12) <= 1e-9


def test_every_modelled_kernel_exists():
    """A model's name is one that the library reports its launches under (the
    FP64 elimination of every interval is kept as a reference count)."""
    src = "".join(open(os.path.join(ROOT, "paper_1507_04769_gb300", "csrc", f)).read()
                  for f in sorted(os.listdir(os.path.join(ROOT, "paper_1507_04769_gb300", "csrc"))))
    text = open(os.path.join(ROOT, "bench.py")).read()
    body = text[text.index("    models = {"):text.index("    peaks_path =")]
    names = [n for n in re.findall(r'^        "(k_\w+)"(?: \+ suffix)?: \(', body, re.M)]
    assert len(names) >= 12
    for n in names:
        if n != "k_condense_smem_fp64":
            assert n + '"' in src or all(n + t + '"' in src for t in ("_fp32", "_fp64")), n
