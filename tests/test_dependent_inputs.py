"""Kernels that start while the kernel in front still runs must not take what that one writes as `const ... __restrict__`: the compiler may
fetch such data through the read-only path, which griddepcontrol.wait does not order.  What may be is listed here: constants of the model,
of a tree and of a step's call, and, per kernel, what is at least two kernels old (read ahead of the wait on purpose)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_13344_b200", "csrc")
CONSTANTS = {"W", "embed", "gain", "rope", "page_table", "parent", "depth", "anc", "head_of", "rank_of", "kper", "plant"}
OLDER = {"rope_append_kernel": {"len", "n_active", "row_off"}, "topk_merge_kernel": {"root"}}


def test_no_dependent_kernel_takes_its_inputs_as_read_only():
    seen, wrong = set(), []
    for name in sorted(os.listdir(CSRC)):
        src = open(os.path.join(CSRC, name)).read()
        for m in re.finditer(r"__global__ void\s*(?:__launch_bounds__\([^;{]*?\)\s+)?(\w+)\(([^{]*?)\)\s*\{", src):
            kernel, params = m.groups()
            body = src[m.end():]
            body = body[:body.index("\n}")]
            if "griddep_wait()" not in body:
                continue
            seen.add(kernel)
            read_only = set(re.findall(r"const \w+\s?\* ?__restrict__ (\w+)", params))
            wrong += [(name, kernel, p) for p in sorted(read_only - CONSTANTS - OLDER.get(kernel, set()))]
    assert {"row_norm_kernel", "argmax_rows_kernel", "gemm_f32_small_kernel", "accept_kernel", "tree_attn_f32_kernel", "swiglu_kernel",
            "fused_norm_kernel", "gate_kernel", "kv_compact_kernel", "topk_merge_kernel", "head_init_kernel"} <= seen
    assert not wrong
