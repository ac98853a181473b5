"""Kernels whose launches may overlap (launch_next) start while earlier kernels of the
chain still write: none may take those data through a const __restrict__ parameter,
which promises that they stay as they are for the kernel's lifetime. What goes wrong
otherwise cannot show in the rates (the positions so read decide pairs at the cutoff,
where the kernel is zero), so the rule is checked in the sources."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1904_00861_gb300", "csrc")


def test_no_overlapping_kernel_promises_constant_inputs():
    text = {f: open(f).read() for f in sorted(glob.glob(os.path.join(CSRC, "*.cu")))}
    names = {n for t in text.values() for call in re.findall(r"launch_next\((?!const)[^;]*;", t)
             for n in re.findall(r"\bk_\w+", call)}
    assert {"k_bin_keys", "k_scatter", "k_rank_move", "k_nlist_home", "k_nlist_cells2", "k_state_n", "k_rates_out"} <= names
    for name in names:
        found = [m for t in text.values() for m in re.findall(r"__global__[^;{]*?\b%s\(([^)]*)\)\s*\{\s*(.*?);" % name, t, re.S)]
        assert len(found) == 1, name
        params, first = found[0]
        assert first.startswith("grid_start<"), name
        for p in params.split(","):
            assert not re.search(r"\bconst\b.*__restrict__", p), (name, p)
