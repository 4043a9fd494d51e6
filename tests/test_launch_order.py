"""Order of dependent kernels (no GPU): every kernel is launched with programmatic
stream serialisation, so what keeps the stream's order is where each kernel calls
pdl_wait() and pdl_trigger().  A wrong place shows only as a rare race, so the
sources are checked: by kernel, the statements in front of the first wait."""
import glob
import os
import re

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2608_28099_gb300", "csrc")


def _kernels():
    """name -> body of every __global__ function, comments removed."""
    out = {}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        with open(path) as f:
            s = re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", f.read(), flags=re.S))
        for m in re.finditer(r"__global__\s+void\b.*?(\w+)\s*\((?=\s*(?:const\s+)?(?:__grid_constant__|"
                             r"T\b|TX\b|float\b|float4\b|PartIn\b|QkvRopeArgs\b|AttnArgs\b|CUtensorMap\b))", s, flags=re.S):
            i = s.index("{", m.end())
            depth, j = 1, i + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(s[j], 0)
                j += 1
            out[m.group(1)] = s[i:j]
    return out


KERNELS = _kernels()

# Blocks that may leave before the wait, since others of the same grid always wait
# (a grid is complete only when all of its blocks are).
LEAVES_EARLY = {
    "attn_tc_kernel": "groups past the last share; group 0 has one",
    "attn_tok_kernel": "groups past the last share; group 0 has one",
    "attn_split_simt": "units past the sequence's end; unit 0 never is (k >= 1 new rows)",
}


def test_every_kernel_is_found():
    with_launch = set()
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        with open(path) as f:
            with_launch |= set(re.findall(r"launch_k\(\s*(\w+)", f.read()))
    assert with_launch == set(KERNELS)


@pytest.mark.parametrize("name", sorted(KERNELS))
def test_a_grid_completes_after_the_one_before_it(name):
    body = KERNELS[name]
    assert "pdl_wait()" in body, "a grid that never waits may complete before the one in front of it"
    before = body[:body.index("pdl_wait()")]
    if name not in LEAVES_EARLY:
        assert not re.search(r"\breturn\b", before), "a block leaves before the wait"


# The kernels that can be the first of a public call: per-sequence rows and hidden
# states start with the input norm, the shared prompt with the rotation, sp_attend on
# CUDA cores with the split kernel (on tensor cores a memset is in front), sp_project
# with the conversion of X or, on CUDA cores, with its only kernel.
FIRST = ["rmsnorm_rows_kernel", "rmsnorm_rows_loop_kernel", "qkv_rope_kernel", "qkv_rope_rows_kernel",
         "attn_split_simt", "to_act_kernel"]
ALONE = ["gemm_simt_kernel", "gemv_simt_kernel"]


@pytest.mark.parametrize("name", FIRST)
def test_a_first_kernel_triggers_after_its_wait(name):
    # kernels behind it read the caller's ids, lengths, page table, cache and weights
    # in front of their own waits
    body = KERNELS[name]
    assert body.index("pdl_wait()") < body.index("pdl_trigger()")


@pytest.mark.parametrize("name", FIRST + ALONE)
def test_a_first_kernel_reads_the_callers_data_after_its_wait(name):
    before = KERNELS[name]
    before = before[:before.index("pdl_wait()")]
    assert not re.search(r"resolve_seq|load_tile\(|load4\(|load8\(|\bx\[|\bX\[|\bW\[|xr\b", before)


def test_readout_lanes_fence_between_the_count_and_the_other_blocks_partials():
    # one lane counts the block; every lane of the last block reads partials that
    # other blocks wrote, so each needs its own fence after it learns the verdict
    body = KERNELS["readout_kernel"]
    after = body[body.index("__shfl_sync(0xffffffffu, is_last"):]
    before_reads = after[:after.index("__ldcg(")]
    assert "__syncwarp()" in before_reads and "__threadfence()" in before_reads


def test_both_ctas_of_a_pair_wait_for_what_arrives_on_their_barriers():
    # a commit of the pair arrives on the barrier of both CTAs; one that left before
    # the arrival landed would have it written into the next block's shared memory
    body = KERNELS["gemm_pair_kernel"]
    end = body[body.rindex("__syncthreads()"):]
    assert re.search(r"rank\s*!=\s*0\s*\)\s*mbar_wait_drain\(fin\b", end[:end.index("cluster_sync()")])
