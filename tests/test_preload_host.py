"""The first call of the fixed-scratch step loads every kernel that its launch chain can reach (read off the sources: whether a
kernel's code is loaded cannot be asked without loading it)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2504_05295_b200", "csrc")

# launched by other entry points only, or for shapes beyond the built-in array
ELSEWHERE = {
    "k_set_scalar": "graph replay of dion_step",
    "k_copy_chain": "chains", "k_form_b32_chain": "chains", "k_round_f16_chain": "chains", "k_round_tf32_chain": "chains",
    "k_split_bf16_chain": "chains", "k_colsumsq_finish": "sharded calls",
    "k_range_partial": "M + G in scratch", "k_form_sum_amax": "M + G in scratch", "k_split_sum": "M + G in scratch", "k_split_f16_fixed": "M + G in scratch",
    "k_absmax_partial": "panels of 2e9 operations", "k_split_f16_scaled": "panels of 2e9 operations",
    "k_split_f16_tri": "panels of 2e9 operations", "k_near_identity": "panels of 2e9 operations",
    "k_near_end": "panels of 2e9 operations",
}


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def body(text, head):
    start = text.index(head)
    return text[start:text.index("\n}", start)]


def test_first_call_loads_what_the_step_launches():
    api = source("dion_api.cu")
    launched = set(re.findall(r"launch_pdl\((k_\w+)|\(const void\*\)(k_\w+)|\b(k_\w+)(?:<\w+>)?<<<", api))
    launched = {name for names in launched for name in names if name}
    loaded = set(re.findall(r"touch_kernel\((k_\w+)", body(api, "bool preload_kernels()")))
    assert launched > {"k_copy_block", "k_chol_flow", "k_hh_apply"}
    assert launched - loaded - set(ELSEWHERE) == set()
    assert set(ELSEWHERE) <= launched


def test_first_call_loads_every_instance_of_a_template():
    # (also those that a helper launches for its caller: go(...))
    api = source("dion_api.cu")
    named = lambda text, call: {re.sub(r"\s", "", k) for k in re.findall(call + r"\((k_\w+(?:<[^>]*>)?)", text)}
    launched = named(api, r"(?:launch_pdl|\bgo)")
    assert {"k_probe_fused<true>", "k_probe_fused<false>", "k_gemm_simt<64,64,16,4,4,2,GemmSecond>"} <= launched
    missing = launched - named(body(api, "bool preload_kernels()"), "touch_kernel")
    assert {k for k in missing if k.split("<")[0] not in ELSEWHERE and "GemmTabs" not in k} == set()      # (GemmTabs: chains)


def test_the_tensor_engine_loads_its_own_reduction():
    # a static kernel of a header is one kernel per translation unit
    umma = source("umma_gemm.cuh")
    assert re.search(r"static __global__ void k_splitk_reduce", source("simt_gemm.cuh"))
    assert re.search(r"cudaLaunchKernelEx\(&cfg, k_splitk_reduce", umma)
    assert "k_splitk_reduce" in body(umma, "int umma_configure()")
