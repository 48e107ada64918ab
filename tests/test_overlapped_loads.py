"""Kernels that are launched overlapped (they call grid_wait) may start before the kernel ahead of them has ended.

Data that no kernel of such a chain writes may come through the non-coherent path (__ldg, or a const __restrict__
argument); the states, scales and digits that one kernel of the chain hands to the next may not."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1309_5994_gb300", "csrc")
# written before a chain starts and not by its kernels
CONSTANT = {"src_site", "src_time", "I.nbr", "I.nbond", "I.rsrc", "I.adown", "Jz", "Jtab", "nbr", "nbond", "lam", "esig",
            "as", "scale", "rref", "map_hi", "map_lo"}


def _kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for part in text.split("__global__")[1:]:
            if "grid_wait()" in part.split("\n}\n")[0]:
                yield os.path.basename(path), part.split("\n}\n")[0]


def test_chain_data_is_read_by_ordinary_loads():
    seen = set()
    for path, body in _kernels():
        name = re.search(r"(k_\w+)\s*\(", body).group(1)
        seen.add(name)
        head, code = body.split("{", 1)
        for arg in re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", head):
            # xs: slices, read by bulk copies only
            assert arg in CONSTANT or arg in ("xs", "run", "sweeps_done"), (name, arg)
        for arg in ("run", "sweeps_done"):
            for use in re.findall(r"[^\n]*\*[^\n;]*\b%s\b(?!->)[^\n]*" % arg, code):
                assert "volatile" in use or "(" + arg not in use.replace(" ", ""), (name, use)
        for src in re.findall(r"__ldc?[sg]\(\s*(?:reinterpret_cast<const float4\*>\()?\(?&?([\w.]+)", code):
            assert src in CONSTANT, (path, name, src)
    assert seen == {"k_oz64_xprep", "k_oz64_gemm", "k_f64_check", "k_series_check", "k_tc_fused"}


def test_the_fused_epilogue_reads_the_state_by_ordinary_loads():
    text = open(os.path.join(CSRC, "k_tc.cu")).read()
    body = text[text.index("struct FusedEpilogue {"):text.index("__device__ __forceinline__ bool r_is_zero")]
    assert "__ldcs(din" not in body and "__ldg(" not in body and "__restrict__ din" not in body
