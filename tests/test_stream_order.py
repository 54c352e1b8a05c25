"""Work on a context's memory is ordered by the stream that uses it.

The solver's own stream, and a stream that a caller passes, are non-blocking: neither
waits for the default stream.  A clear or a copy on the default stream is therefore not
ordered before the kernels that follow it, and the fault shows only on large arrays.  The
CPU tests read the sources for such calls; the GPU tests run starts that the fault reaches.
"""
import re
from pathlib import Path

import numpy as np
import pytest
import torch

import paper_2407_15049_gb300 as L
import workloads as W

CSRC = Path(L.__file__).resolve().parent / "csrc"


def _body(name: str, head: str) -> str:
    """Text of the function whose definition starts with `head` (up to the next closing brace in
    column 0)."""
    text = (CSRC / name).read_text()
    at = text.index(head)
    return text[at:text.index("\n}", at)]


@pytest.mark.parametrize("name,head", [
    ("api.cu", "lorads_status alloc_state("),
    ("api.cu", "lorads_status admm_alloc("),
    ("gnn.cu", 'extern "C" lorads_status lorads_gnn_create('),
    ("gnn.cu", 'extern "C" lorads_status lorads_gnn_set_params('),
])
def test_clears_and_copies_name_their_stream(name, head):
    body = _body(name, head)
    assert not re.search(r"\bcuda(Memset|Memcpy)\(", body)


def test_iteration_limit_of_a_batch_is_set_on_its_stream():
    body = _body("batch.cu", "lorads_status set_iter_limit(")
    assert not re.search(r"\bcudaMemcpy\([^;]*HostToDevice", body)


@pytest.mark.parametrize("name,head,last", [
    ("api.cu", "lorads_status validate_and_build(", "upload("),
    ("batch.cu", 'extern "C" lorads_status lorads_batch_create(', "cudaMemcpyHostToDevice"),
])
def test_uploads_end_before_the_call_returns(name, head, last):
    """A copy from pageable memory on the default stream may return before it ends: the call
    waits for that stream after its last one."""
    body = _body(name, head)
    assert body.rfind("cudaStreamSynchronize(cudaStreamLegacy)") > body.rfind(last) > 0


def _first_iterations(inst, R0, on_device, stream, prec, iters):
    ctx = L.lorads_create(inst, L.default_params(prec=prec, lbfgs_mem=2), stream=stream.cuda_stream)
    try:
        res = L.lorads_solve(ctx, R0, on_device=on_device, max_total_inner=iters)
        R, y = L.lorads_get_solution(ctx, inst.n, inst.m)
    finally:
        L.lorads_destroy(ctx)
    return res["inner_iters"], R, y


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [L.LORADS_MIXED, L.LORADS_FP64])
def test_first_solve_on_a_callers_stream_takes_every_start(prec):
    """The first solve of a new context, at a size where clearing the history takes longer than
    the host needs to start the copy: pinned and pageable host starts give the bits of the
    start that lies on the device."""
    n, r = 2000000, 24
    inst = W.maxcut_instance(n, W.er_graph(n, n, 1, "pm1"))
    stream = torch.cuda.Stream()
    gen = torch.Generator(device="cuda").manual_seed(5)
    R0 = torch.randn(n, r, generator=gen, dtype=torch.float64, device="cuda")
    R0 /= R0.norm(dim=1, keepdim=True)
    host = R0.cpu()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        want = _first_iterations(inst, R0, True, stream, prec, 2)
        for start in (host.pin_memory().numpy(), host.numpy()):
            got = _first_iterations(inst, start, False, stream, prec, 2)
            assert got[0] == want[0]
            assert np.array_equal(got[1], want[1]) and np.array_equal(got[2], want[2])
