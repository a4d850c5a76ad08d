"""The Laplace kernels that are launched while their producer still runs (those that
call lap_wait_previous) take no buffer of that producer as a restricted pointer:
const __restrict__ declares its data unchanged for the kernel's lifetime, and a
load of it may then be moved before the wait.  Read from the source (CPU)."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1606_03255_gb300", "csrc",
                   "fl_laplace.cu")
PRODUCED = {"partial", "u", "ha", "g"}      # written by the kernels of the same call


def test_dependent_kernels_take_no_produced_buffer_as_restricted():
    text = open(SRC, encoding="utf-8").read()
    kernels = re.findall(r"__global__\s+void(?:\s+__launch_bounds__\([^)]*\))?\s+(k_\w+)\(([^)]*)\)\s*\{([^\n]*\n[^\n]*)",
                         text)
    dependents = {name: params for name, params, head in kernels if "lap_wait_previous()" in head}
    assert set(dependents) == {"k_lap_reduce_items", "k_lap_couple_cheb", "k_lap_eval_cheb", "k_gen_eval"}
    for name, params in dependents.items():
        for prm in params.split(","):
            word = re.search(r"(\w+)\s*$", prm).group(1)
            assert not (word in PRODUCED and "__restrict__" in prm), (name, prm.strip())
