"""Kernels launched as programmatic dependents start while the kernel before them writes,
so they may read what it writes only by plain loads after their wait: the non-coherent path
(__ldg, or a const __restrict__ parameter) is for data that nobody writes during the
kernel's life.  A race of this kind shows in no result, so the sources are checked."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_05583_gb300", "csrc")
SOURCES = {os.path.basename(p): open(p).read() for p in glob.glob(os.path.join(CSRC, "*.cu*"))}

# Parameters that the kernel before may still be writing.
WRITTEN_BEFORE = {
    "k_to_row_major": ["srcT"],
    "k_to_row_major_wide": ["srcT"],
    "k_grad_reduce": ["ws_s", "ws_r", "ws_j"],
    # First kernels of a call: every input may be another call's output.
    "k_decode_tile": ["x_t", "coef"],
    "k_decode_any": ["x_t", "coef"],
    "k_decode_coupled": ["x_t", "coef", "c_raw"],
    "k_mixer_finish": ["x_t", "g_t", "z_t", "hist", "conv_w", "scale", "c_raw"],
    "k_conv_tail": ["hist"],
}
# Kernels that read earlier results through a structure's plain pointers or bulk copies.
THROUGH_STRUCTURES = {"k_scan", "k_backward_tc", "k_terminal_tc", "k_mixer_stream"}


def kernel(name):
    """(parameter list, body) of a __global__ function."""
    for src in SOURCES.values():
        m = re.search(r"__global__ void (?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?" + name + r"\(", src)
        if m:
            end = src.index(") {", m.end())
            depth, i = 1, end + 3
            while depth:
                depth += {"{": 1, "}": -1}.get(src[i], 0)
                i += 1
            return src[m.end():end], re.sub(r"//[^\n]*", "", src[end + 3:i])
    raise AssertionError(f"no kernel {name}")


def dependent_kernels():
    names = set()
    for src in SOURCES.values():
        for m in re.finditer(r"(?:launch_dependent|launch_pdl|launch_pdl_block|cudaLaunchKernelEx)\(\s*(?:&cfg,\s*)?(\w+)", src):
            names.add(m.group(1))
        # A launcher that takes the kernel as an argument.
        names.update(re.findall(r"\bgo\((k_\w+)", src))
        names.update(re.findall(r"auto \*k = (k_\w+)", src))
    return {n for n in names if n.startswith("k_")}


def test_every_dependent_kernel_is_listed():
    assert dependent_kernels() == set(WRITTEN_BEFORE) | THROUGH_STRUCTURES


@pytest.mark.parametrize("name", sorted(WRITTEN_BEFORE) + sorted(THROUGH_STRUCTURES))
def test_dependent_kernels_wait(name):
    body = kernel(name)[1]
    assert "pdl_wait()" in body or "griddepcontrol.wait" in body


@pytest.mark.parametrize("name", sorted(WRITTEN_BEFORE))
def test_results_of_the_kernel_before_are_read_by_plain_loads(name):
    params, body = kernel(name)
    assert "__ldg(" not in body
    for p in params.split(","):
        ident = re.search(r"(\w+)\s*$", p.strip()).group(1)
        if ident in WRITTEN_BEFORE[name]:
            assert not ("const" in p and "__restrict__" in p), p.strip()


def test_helpers_of_dependent_kernels_use_plain_loads():
    assert "__ldg(" not in SOURCES["rlm_device.cuh"].replace("__ldg() (which", "")
    assert "__ldg(" not in SOURCES["rlm_mixer.cuh"]
    mix = SOURCES["rlm_decode.cu"]
    assert "__ldg(" not in mix[mix.index("MixPart<T> mix_part("):mix.index("void mix_shift(")]


# Decode steps are the first kernel of their call and a dependent launch: the kernel before
# them may write anything they read.
@pytest.mark.parametrize("name", ["k_decode_tile", "k_decode_any", "k_decode_coupled", "k_mixer_finish"])
def test_decode_kernels_read_nothing_before_their_wait(name):
    params, body = kernel(name)
    before = re.split(r"pdl_wait\(\)|griddepcontrol\.wait", body)[0]
    before = re.sub(r"prefetch_\w+\([^;]*;", "", before)
    pointers = [re.search(r"(\w+)\s*$", p.strip()).group(1) for p in params.split(",") if "*" in p]
    for p in pointers + ["mix.hist", "mix.conv_w", "mix.scale"]:
        assert not re.search(r"(?<![\w.])" + re.escape(p) + r"\b", before), f"{p} is used before the wait"
