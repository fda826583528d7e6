"""The surrogate kernel's two groups of warps meet at named barriers only."""
import os
import re

import numpy as np
import pytest
import torch

import oracle
from paper_2202_10647_gb300 import ionize, workloads as W

CSRC = os.path.join(os.path.dirname(os.path.abspath(ionize.__file__)), "csrc")


def test_no_block_barrier_on_a_branch():
    """CUDA defines __syncthreads and its variants only where the whole block
    reaches the same call: none may stand in the branch of the network warps
    or in that of the cell warps."""
    src = open(os.path.join(CSRC, "surrogate.cu")).read()
    src = re.sub(r"//[^\n]*", "", src)
    a = src.index("if (t < kM) {")
    depth, i = 0, a
    while True:  # to the end of the else branch
        if src[i] == "{":
            depth += 1
        elif src[i] == "}":
            depth -= 1
            if depth == 0 and not src[i + 1:].lstrip().startswith("else"):
                break
        i += 1
    branches = src[a:i]
    assert "bar_sync<kBarYFree" in branches and "wait_outputs" in branches
    assert "__syncthreads" not in branches


@pytest.mark.gpu
def test_tiles_the_network_skips():
    """All cells by the network kernel, with runs of 128-cell tiles none of
    whose cells it could serve between tiles that it serves: both groups
    take the same tiles, and every cell is stepped."""
    from test_gpu_step import check, gpu_species, oracle_species
    from test_gpu_surrogate import rand_P

    sd = W.argon_like()
    l2lo, l2hi = np.log2(10.0), np.log2(1e5)
    norm = {"log2E_min": float(l2lo), "log2E_max": float(l2hi), "y_floor": -40.0,
            "y_mean": [0.0] * sd.Z, "y_scale": [1.0] * sd.Z}
    P = torch.tensor(rand_P(sd.Z, 11, 0.3), dtype=torch.float32, device="cuda")
    net = ionize.Surrogate(gpu_species(sd), P, norm)
    n = 128 * 1500 + 77
    wl = W.ladder_cells(sd, n, 46, block=64)
    tile = torch.arange(n) // 128
    E = wl.E.clone()
    off = (tile * 7 % 11 < 6) | (tile // 100 % 3 == 1)
    E[off] = 3.0  # below the trained range
    E[off & (torch.arange(n) % 5 == 0)] = 2.0e5
    lo, hi, N = wl.lo.cuda(), wl.hi.cuda(), wl.N.cuda()
    dne = torch.full((n,), float("nan"), device="cuda")
    ws = net.step(E.cuda(), N, lo, hi, 0.05, dne, pop_tol=1e-30)  # never trusted, always asked
    torch.cuda.synchronize()
    assert ionize.surrogate_counters(ws) == (0, n, 0)
    No, loo, hio, dneo = oracle.step(oracle_species(sd), E.double().numpy(),
                                     wl.N[:, :n].double().numpy(), 0.05, wl.lo.numpy(),
                                     wl.hi.numpy())
    out = dict(N=N.double().cpu().numpy(), lo=lo.cpu().numpy(), hi=hi.cpu().numpy(),
               dne=dne.double().cpu().numpy())
    check(out, dict(N=No, lo=loo, hi=hio, dne=dneo), wl.lo, wl.hi, ionize.ION_F32, n=n, sd=sd,
          E=E.double().numpy())
