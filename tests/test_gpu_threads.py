"""The entry points called from threads that have made no CUDA call before."""
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu


def _in_a_new_thread(f):
    out = []

    def run():
        try:
            out.append(f())
        except Exception as e:                             # noqa: BLE001 - handed to the caller
            out.append(e)

    t = threading.Thread(target=run)
    t.start()
    t.join()
    if isinstance(out[0], Exception):
        raise out[0]
    return out[0]


@pytest.mark.parametrize("code", [(2, 2), (2, 13), (2, 53)])
@pytest.mark.parametrize("batch", [1, 33])
def test_products_from_a_new_thread(code, batch):
    import paper_2603_11021_b200 as P
    ctx, n_out, k_in = P.Context(*code, device=0), 256, 480
    nblocks = n_out * (k_in // 24)
    stream = torch.zeros(ctx.index_bytes(nblocks), dtype=torch.uint8, device="cuda")       # field 0: the point (4, 4, 0, ..)
    gain = torch.full((nblocks,), 0.25, dtype=torch.half, device="cuda")
    x = torch.ones((batch, k_in), dtype=torch.bfloat16, device="cuda")
    gemm, gemv = P.llvq_sort_blocks_gemm(ctx, stream, n_out, k_in), P.llvq_sort_blocks(ctx, stream, n_out, k_in)
    y, yb = torch.empty(n_out, device="cuda"), torch.empty((batch, n_out), dtype=torch.bfloat16, device="cuda")
    torch.cuda.synchronize()                               # the threads launch on streams of the same context one after the other
    calls = {"gemm": lambda: P.llvq_gemm_small_batch(ctx, stream, gain, n_out, k_in, x, yb),
             "gemm_sorted": lambda: P.llvq_gemm_small_batch_sorted(ctx, gemm, gain, n_out, k_in, x, yb),
             "gemm_noalloc": lambda: P.llvq_gemm_small_batch_noalloc(ctx, stream, gain, n_out, k_in, x, yb),
             "gemv": lambda: P.llvq_gemv(ctx, stream, gain, n_out, k_in, x[0], y),
             "gemv_sorted": lambda: P.llvq_gemv_sorted(ctx, gemv, gain, n_out, k_in, x[0], y),
             "dequant": lambda: P.llvq_dequant_matrix(ctx, stream, gain, n_out, k_in, P.LLVQ_LAYOUT_ROWWISE).float().sum(1)}
    for name, call in calls.items():
        y.fill_(-1.0), yb.fill_(-1.0)
        torch.cuda.synchronize()
        got = _in_a_new_thread(call)
        torch.cuda.synchronize()
        assert (got.float() == 2.0 * (k_in // 24)).all(), name
    assert P.llvq_last_error(ctx) == (0, 0)


def test_first_launches_of_a_context_inside_a_capture():
    # the kernels have been launched before, by another context: what the host settles for a new one is no work on the stream
    import paper_2603_11021_b200 as P
    n_out, k_in, batch = 256, 480, 16
    nblocks = n_out * (k_in // 24)
    gain = torch.full((nblocks,), 0.25, dtype=torch.half, device="cuda")
    x = torch.ones((batch, k_in), dtype=torch.bfloat16, device="cuda")
    y, yb = torch.empty(n_out, device="cuda"), torch.empty((batch, n_out), dtype=torch.bfloat16, device="cuda")
    for capture in (False, True):
        ctx = P.Context(2, 13, device=0)
        stream = torch.zeros(ctx.index_bytes(nblocks), dtype=torch.uint8, device="cuda")
        y.fill_(-1.0), yb.fill_(-1.0)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        if capture:
            with torch.cuda.graph(graph):
                P.llvq_gemv(ctx, stream, gain, n_out, k_in, x[0], y)
                P.llvq_gemm_small_batch(ctx, stream, gain, n_out, k_in, x, yb)
            graph.replay()
        else:
            P.llvq_gemv(ctx, stream, gain, n_out, k_in, x[0], y)
            P.llvq_gemm_small_batch(ctx, stream, gain, n_out, k_in, x, yb)
        torch.cuda.synchronize()
        assert (y == 2.0 * (k_in // 24)).all() and (yb.float() == 2.0 * (k_in // 24)).all()
        assert P.llvq_last_error(ctx) == (0, 0)
        del graph
