"""Kernels that may start before the kernel in front of them has finished (those that call
pdl_wait) read nothing through the read-only path: its contract is that nobody writes the
data while the kernel lives, and the kernel in front may still be writing it."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2609_18145_gb300", "csrc")

# the GEMM's bias is a parameter and its aux the activations of the forward pass: the kernel
# in front of it writes neither
ALLOWED = {("gemm_pair_kernel", "__ldg")}


def kernels(text):
    """(name, signature and body) of every __global__ function of a source."""
    text = re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)
    for m in re.finditer(r"__global__\s+void\b", text):
        start = text.index("{", m.end())
        depth, i = 0, start
        while True:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
            if depth == 0:
                break
        head = re.sub(r"__launch_bounds__\s*\((?:[^()]|\([^()]*\))*\)", "", text[m.end():start])
        yield re.search(r"(\w+)\s*\(", head).group(1), text[m.start():i]


def test_dependent_kernels_stay_off_the_read_only_path():
    found = set()
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        for name, body in kernels(open(path).read()):
            if "pdl_wait()" not in body:
                continue
            found.add(name)
            for word in ("__restrict__", "__ldg", "ld.global.nc"):
                if (name, word) in ALLOWED:
                    continue
                assert word not in body, (name, word)
    # the scan sees the kernels it is about
    assert {"hcw_tc_kernel", "hcw_dwp_kernel", "hcw_small_kernel", "decode_mma_kernel",
            "gemm_pair_kernel", "f32_fwd_kernel", "f32_dx_kernel", "f32_dw_kernel",
            "f32_chain_kernel", "relu_grad_kernel", "splitk_reduce_kernel"} <= found
