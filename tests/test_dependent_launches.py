"""Kernels launched with a programmatic dependency start while the kernel before
still writes what they read after their wait.  A `const ... __restrict__`
parameter tells the compiler that nothing writes the data while the kernel runs
(it may then load it early, or through the read-only path), so these kernels
take none but for data that was complete before the kernel before started (not
gpu)."""
import glob
import os
import re

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2603_04035_gb300", "csrc")
# launched through a variable
OTHERS = {"mlp_gemm_kernel", "mlp_layer_kernel", "epoch_force_kernel"}
# written before the kernel before started: the previous step's weights and rows; F2's derivative, the head in between
OLDER = {"mlp_head_loss_kernel": {"W3f", "P", "rows"}, "mlp_l3back_kernel": {"W3f", "dgelu2"}}


def test_dependent_kernels_promise_nothing_about_what_they_read():
    src = {os.path.basename(p): re.sub(r"//[^\n]*", "", open(p).read()) for p in glob.glob(os.path.join(CSRC, "*.cu*"))}
    names = set(OTHERS)
    for text in src.values():
        # launch_dep(c, kernel, grid, block, shared memory, dependent, ...)
        calls = re.findall(r"launch_dep\(\s*c\s*,\s*(\w+_kernel)(?:<\w+>)?\s*,((?:[^(),]|\((?:[^()]|\([^()]*\))*\)|,)*)", text)
        for name, args in calls:
            rest = re.sub(r"\([^()]*(?:\([^()]*\)[^()]*)*\)", "", args).split(",")
            if rest[3].strip() != "false":
                names.add(name)
    assert {"pca_cmul_kernel", "pca_gram_kernel", "mlp_head_loss_kernel", "mlp_l3back_kernel"} <= names
    promise = re.compile(r"\bconst\b[^,;]*\*\s*__restrict__")
    bad = []
    for name in sorted(names):
        (params,) = [m for text in src.values() for m in re.findall(r"__global__[^;{]*?\b" + name + r"\s*\(([^{]*?)\)\s*\{", text)]
        bad += [f"{name}: {' '.join(p.split())}" for p in params.split(",")
                if promise.search(p) and p.split()[-1] not in OLDER.get(name, ())]
    # the epochs' positions, the one member of a by-value structure that a kernel before writes
    (args,) = re.findall(r"struct EpochArgs \{(.*?)\n\};", src["epoch.cuh"], flags=re.S)
    bad += [line.strip() for line in args.split("\n") if promise.search(line) and "Y_in" in line]
    assert not bad, "\n".join(bad)
