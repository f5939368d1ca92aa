"""What a pass of the smoother kernel writes to global memory and a later pass of
the same launch reads by bulk copies: the copies go through another proxy than the
stores, so every writing lane has to fence after its last store. A missing fence
shows in no result on most runs, so the order is checked in the source here, and on
the GPU by runs whose first copy is of the step written last. The same for the exit
of the iterations' loop, which all of a block's threads have to take together."""
import os
import re

import numpy as np
import pytest
import torch

from paper_2102_00514_gb300 import build, pes, synth

KERNEL = os.path.join(build.CSRC, "pes_kernel.cuh")
FENCE = "stores_before_bulk_reads();"


def body(name):
    """Source of the function template `name`, from its signature to its closing brace."""
    src = open(KERNEL).read()
    at = re.search(r"PES_DEV bool %s\(" % name, src).start()
    return src[at:src.index("\n}\n", at)]


@pytest.mark.parametrize("name,stores", [("fold_filter_chunk", ("store_lin_obs<K>(", "store_lin_trans<K>(")),
                                         ("rerun_filter_chunk", ("store_xP(",))])
def test_stores_are_fenced_before_the_pass_returns(name, stores):
    code = body(name)
    last = max(code.rindex(s) for s in stores)
    assert FENCE in code[last:], f"{name}: stores that a later pass streams are not fenced"


def test_blocks_leave_the_iterations_as_one():
    """The status word can change while a block's warps read it; a loop exit taken
    by some of them only would leave the others at barriers without them."""
    src = open(KERNEL).read()
    loop = src[src.index("for (it = 0; it < p.iters; ++it) {"):]
    exit_line = next(l for l in loop.splitlines() if "p.status" in l and "break;" in l)
    assert "__syncthreads_or(" in exit_line


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [pes.FP64, pes.FP32])
@pytest.mark.parametrize("method", [pes.IEKS, pes.CUBATURE, pes.GAUSS_HERMITE])
def test_runs_repeat_bit_for_bit(method, prec):
    """Short chunks: the RTS pass starts with the step that the re-run wrote last.
    Sums have a fixed order, so repeated runs are equal to the bit."""
    dt = torch.float64 if prec == pes.FP64 else torch.float32
    with torch.no_grad():
        for T in (61, 500, 4000):
            wl = synth.ct_bearings([T], seed=T, sensor_jitter=0.2, omega0_halfwidth=1.0)
            dev = lambda a, t=dt: torch.as_tensor(np.ascontiguousarray(a), dtype=t, device="cuda")
            args = (pes.Model.from_workload(wl), method, prec, dev(wl["y"]), dev(wl["offsets"], torch.int64),
                    dev(wl["m0"]), dev(wl["P0"]))
            sm = pes.Smoother(T + 1, 1)
            x0, P0, _, _ = sm.ieks_run(*args, iters=3)
            assert torch.isfinite(x0).all()
            for _ in range(20):
                x, P, _, _ = sm.ieks_run(*args, iters=3)
                assert torch.equal(x, x0) and torch.equal(P, P0), T
            sm.close()
