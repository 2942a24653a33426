"""The statistics kernel runs on a cluster whose blocks write into the first block's shared memory:
none may do so before that block is known to run.  By reading: a barrier of the cluster stands
before the first write; on the GPU: small sets, whose blocks reach that write at once, give the
same statistics at every launch while another stream keeps the SMs busy."""
import os
import re

import pytest
import torch

from paper_2609_32920_gb300 import build, lt


def test_cluster_barrier_before_remote_shared_memory():
    src = open(os.path.join(build.CSRC, "lt_mlp.cu")).read()
    src = re.sub(r"//[^\n]*", "", src)
    kernels = [k for k in re.split(r"__global__", src)[1:] if "map_shared_rank" in k]
    assert kernels
    for k in kernels:
        first = k.index("map_shared_rank")
        assert "cluster.sync()" in k[:first], "remote shared memory before the cluster's first barrier"
        assert "cluster.sync()" in k[first:], "no barrier between the remote writes and their use"


@pytest.mark.gpu
@pytest.mark.parametrize("n", [512, 513, 1024, 4096])
def test_statistics_repeat_under_load(n):
    g = torch.Generator(device="cuda").manual_seed(n)
    X = torch.randn((n, 16), device="cuda", generator=g)
    T = torch.randn(n, device="cuda", generator=g)
    want = torch.zeros(lt.MLP_PARAMS, device="cuda")
    lt.mlp_init_stats(want, X, T)
    outs = [torch.zeros(lt.MLP_PARAMS, device="cuda") for _ in range(64)]
    big = torch.zeros(1 << 24, device="cuda")
    other = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(other):
        for _ in range(64):
            big.add_(1.0)
    for P in outs:
        lt.mlp_init_stats(P, X, T)
    torch.cuda.synchronize()
    # FP64 atomic sums: their order may move the last bit of the rounded FP32 result
    for P in outs:
        assert torch.allclose(P, want, rtol=1.2e-7, atol=1e-9)
