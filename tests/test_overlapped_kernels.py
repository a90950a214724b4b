"""Kernels launched with programmatic overlap start while the kernel before them still writes their operands: their sources may
not promise the compiler that those do not change."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_14959_b200", "csrc")
SOURCES = {f: open(os.path.join(CSRC, f)).read() for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cuh"))}

#: operands that are constant while any forward runs: weights, adapter tables, the routing plan
CONSTANT = re.compile(r"^(reinterpret_cast<const \w+\*>\()?"
                      r"(args\.(bias|ln_g|ln_c1|ln_c2|tile_nslabs|tile_slab|tile_scale|tile_mask|base_wt|hcat)|pos|pos_row|g \+|b \+"
                      r"|\(j < PM_SLAB \? args\.ln_c1 : args\.ln_c2\))")


def overlapped_kernels():
    names = set()
    for text in SOURCES.values():
        for call in re.findall(r"launch_overlapped\(L, (.*?);", text, re.S):
            names |= set(re.findall(r"(\w+_kernel)\b", call))
        if "auto kern" in text and "launch_overlapped(L, kern" in text:
            names |= set(re.findall(r"(select_kernel)<", text))
    return names


def test_the_overlapped_kernels_are_found():
    assert overlapped_kernels() >= {"row_stats_kernel", "heads_kernel", "select_kernel", "plan_upload_kernel", "small_linear_kernel", "shrink_kernel",
                                    "lora_gemm_kernel", "lora_gemm_pair_kernel", "attention_few_kernel", "attention_pipe_kernel",
                                    "attention_tc_kernel"}


def test_their_operands_are_not_declared_invariant():
    for name in overlapped_kernels():
        signatures = [m for text in SOURCES.values() for m in re.findall(r"\b" + name + r"\(([^;{]*?)\)\s*\{", text)]
        assert signatures, name
        for s in signatures:
            assert "__restrict__" not in s, name
    assert "__restrict__" not in re.search(r"void ln_regs\(([^{]*)\{", SOURCES["kernels_simple.cu"]).group(1)


def test_only_constant_operands_are_loaded_as_invariant():
    for name, text in SOURCES.items():
        if name in ("latency_kernel.cu", "contexts.cu"):         # plain launches
            continue
        for operand in re.findall(r"__ldg\((.{0,80})", re.sub(r"//.*", "", text)):
            assert CONSTANT.match(operand), (name, operand)


def test_what_stands_behind_the_routing_plan_is_launched_plainly():
    """The kernels of a forward read the routing plan before they wait for the kernel ahead of them; the kernel that follows the
    plan's writers therefore starts behind their end."""
    overlapped = overlapped_kernels()
    for name in ("im2col_kernel", "latency_forward_kernel", "plan_slots_kernel", "plan_tiles_kernel", "fanout_rows_kernel"):
        assert any(name in text for text in SOURCES.values()) and name not in overlapped, name
    forward = SOURCES["api.cu"][SOURCES["api.cu"].index("int forward_t("):]
    first = re.search(r"CK\((launch_\w+|linear)[<(]", forward).group(1)
    assert first == "launch_im2col"
    upload = SOURCES["plan_device.cu"]
    upload = upload[upload.index("cudaError_t launch_plan_upload"):]
    assert "L.ordered = true;" in upload[:upload.index("\n}\n")]
