"""Kernels that are resident while earlier grids run read what those write by loads that allow for it: ld.global.nc and
__ldg want data that nobody writes while the kernel runs, and neither they nor __ldcg are bound to stay behind a wait."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_02647_b200", "csrc")


def source(path):
    with open(path) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


def test_no_read_only_loads():
    files = glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))
    assert len(files) >= 8
    for f in files:
        src = source(f)
        assert not re.search(r"\.nc\b|\b__ld(g|ca|cg|cs|lu|cv)\(|__restrict__|\btex\dD", src), f
        # loads in assembly are volatile, so that they stay behind the (volatile) wait
        for m in re.finditer(r'asm\s*(volatile)?\s*\(\s*"ld\.global', src):
            assert m.group(1), f


def test_grids_that_wait_first_read_nothing_before():
    """The wait stands before the first access through a pointer of the kernel's parameters."""
    for name, kernel, pointers in (("aggregate.cu", "concat_kernel", r"pp\.[kv]\[|dst\[|kv_pos\[|cu_kv\["),
                                   ("merge.cu", "merge_kernel", r"lse_a\[|lse_b\[|\.load\(|\.store\("),
                                   ("attn_generic.cu", "attn_tiled_kernel", r"p\.kv_len\[|load_tile\(sKV|p\.q_pos\[|kvp\["),
                                   ("prefill_sm100.cu", "prefill_sm100_kernel", r"mbar_init\(q_full")):
        src = source(os.path.join(CSRC, name))
        body = src[re.search(r"__global__[^{;]*\b%s\(" % kernel, src).end():]
        first = re.search(pointers, body)
        assert first and 0 <= body.find("grid_wait();") < first.start(), name
