"""Kernels placed before the ones ahead of them end (grid_begin in csrc/kernels.cuh) read
no other kernel's output through a const __restrict__ pointer, which would let the
compiler load it before the wait: such pointers name the plan's tables only."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2405_14513_gb300", "csrc")
TABLES = {"groups", "rec", "recf", "chunk_lo", "chunk_hi", "bin_chunk", "den"}


def _kernels():
    """(name, parameters, body) of every kernel, and of the device functions they share."""
    for f in ("kernels.cu", "step2_tc.cu", "shell.cu"):
        text = re.sub(r"//[^\n]*|__launch_bounds__[^\n]*", "", open(os.path.join(SRC, f)).read())
        for m in re.finditer(r"(?:__global__|__device__ __forceinline__)[^;{]*?\b(\w+)\(([^{;]*?)\)\s*\{", text):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            yield m.group(1), m.group(2), text[m.end():i]


def test_no_restrict_on_what_kernels_hand_on():
    seen = set()
    for name, params, body in _kernels():
        if "grid_begin()" not in body and name not in ("epi_part", "epi_fin"):
            continue
        seen.add(name)
        read = set(re.findall(r"const\s+[\w:<>\s]+\*\s*__restrict__\s+(\w+)", params))
        allowed = TABLES | ({"in"} if name == "k_fft_z_real" else set())      # an estimate's first kernel
        assert read <= allowed, (name, read - allowed)
    assert {"k_fft_rows_T", "k_ring_gather", "k_fft_cols", "k_step2", "k_step2_tc", "k_reduce", "k_epi_part", "k_epi_fin",
            "k_fft_z_back", "k_ring_scale", "epi_part", "epi_fin"} <= seen, seen
