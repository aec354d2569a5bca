"""The report of the benchmark names the compaction kernel that runs."""

import bench
from paper_2512_02541_b200 import inputs


def test_the_compaction_kernel_of_a_workload():
    def names(wl, n_dropped):
        return bench.compaction_kernels(wl.n_tokens, n_dropped, wl.n_heads, wl.mean_fill)

    wls = inputs.WORKLOADS
    assert names(wls["tiny_n4_g16_s2"], 512) == ["build_kv_small_kernel"]
    assert names(wls["vggt_n800_s9"], 960000) == ["build_kv_stream_kernel", "mean_finalize_kernel"]
    assert names(wls["vggt_n333_s1"], 0) == ["build_kv_gather_kernel"]
    # the few-token kernel's limit: 8,800, 4,400 and 2,200 tokens
    for heads, limit in ((6, 8800), (7, 4400), (18, 4400), (19, 2200)):
        assert bench.compaction_kernels(limit, 1, heads, 2) == ["build_kv_small_kernel"]
        assert bench.compaction_kernels(limit + 1, 1, heads, 0) == ["build_kv_gather_kernel"]
