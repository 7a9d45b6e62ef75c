"""Which kernel serves a linear layer, at sizes on both sides of the rules' lines."""
import pytest
import torch

pytestmark = pytest.mark.gpu

TOKEN_MAJOR, CHANNEL_MAJOR, PAIRS, ROWS = "gemm_i8_kernel", "gemm_i8_t_kernel", "gemm_i8_pair_kernel", "few_rows_kernel"


def _flags(q, kind):
    return {"bf16": q.QDIT_EPI_OUT_BF16, "codes": q.QDIT_EPI_GELU | q.QDIT_EPI_QUANT_OUT, "f32": q.QDIT_EPI_OUT_F32,
            "gated": q.QDIT_EPI_GATE | q.QDIT_EPI_RESIDUAL | q.QDIT_EPI_OUT_BF16}[kind] | q.QDIT_EPI_BIAS


@pytest.mark.parametrize("kind,M,N,K,kernel", [
    # at most 128 rows: half of a pair's tokens would be padding
    ("bf16", 128, 30720, 128, TOKEN_MAJOR), ("bf16", 129, 30720, 128, PAIRS),
    ("codes", 64, 30720, 128, TOKEN_MAJOR), ("gated", 128, 30720, 128, TOKEN_MAJOR), ("gated", 129, 30720, 128, PAIRS),
    # gated layers of more than one wave of token-major tiles: by estimate
    ("gated", 8192, 1152, 1152, CHANNEL_MAJOR), ("gated", 8000, 1152, 4608, CHANNEL_MAJOR), ("gated", 4000, 1160, 1152, PAIRS), ("gated", 65536, 1152, 4608, PAIRS),
    ("gated", 4000, 1160, 64, PAIRS), ("gated", 4096, 1152, 1152, CHANNEL_MAJOR), ("gated", 5000, 3456, 1024, PAIRS),
    # three and four rows of many channels of a short reduction: not streamed
    ("f32", 4, 49152, 752, TOKEN_MAJOR), ("f32", 3, 49152, 768, ROWS), ("f32", 2, 49152, 128, ROWS), ("f32", 3, 16392, 96, TOKEN_MAJOR),
    ("f32", 3, 16392, 80, ROWS), ("f32", 4, 20480, 384, ROWS), ("f32", 4, 16384, 128, ROWS),
    # bf16 output of one wave of channel-major tiles
    ("bf16", 1426, 3072, 4608, CHANNEL_MAJOR), ("bf16", 1024, 4608, 2048, CHANNEL_MAJOR), ("bf16", 1301, 3456, 512, CHANNEL_MAJOR), ("bf16", 1536, 6912, 768, PAIRS), ("bf16", 1024, 2304, 2048, TOKEN_MAJOR),
    # f32 output of many rows: channel-major where the output's own time counts
    ("f32", 2304, 6144, 768, CHANNEL_MAJOR), ("f32", 2304, 6144, 784, PAIRS), ("f32", 1023, 6144, 128, PAIRS),
    ("f32", 2560, 4616, 384, CHANNEL_MAJOR), ("f32", 2560, 4616, 400, PAIRS), ("f32", 3072, 4616, 400, CHANNEL_MAJOR),
    ("f32", 4096, 9216, 1024, CHANNEL_MAJOR), ("f32", 4096, 9208, 1024, PAIRS), ("f32", 1152, 16384, 1152, CHANNEL_MAJOR), ("f32", 1152, 16376, 1152, PAIRS),
    ("f32", 1152, 43688, 1152, CHANNEL_MAJOR), ("f32", 1152, 43696, 1152, PAIRS), ("f32", 2048, 4096, 768, CHANNEL_MAJOR), ("f32", 2048, 4096, 1024, PAIRS),
    ("f32", 1792, 4608, 448, CHANNEL_MAJOR), ("f32", 1792, 4480, 448, PAIRS),
])
def test_route(kind, M, N, K, kernel):
    import paper_2503_02508_b200 as q
    ctx = q.qdit_create(0, None)
    A = torch.ones((M, K), dtype=torch.int8, device="cuda")
    W = torch.ones((N, K), dtype=torch.int8, device="cuda")
    ws, bias, gate = (torch.ones(N, device="cuda") for _ in range(3))
    out = torch.zeros((M, N), dtype={"codes": torch.int8, "f32": torch.float32}.get(kind, torch.bfloat16), device="cuda")
    residual = torch.zeros_like(out)
    epi = q.epilogue(w_scale=ws, bias=bias, gate=gate, ld_gate=N, tokens_per_sample=1 << 20, residual=residual)
    torch.cuda.synchronize()
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        q.qdit_w8a8_linear(ctx, A, W, M, N, K, q.qparams(1.0), None, _flags(q, kind), epi, out, N)
        q.qdit_sync(ctx)
    names = [e.name for e in prof.events() if "_kernel" in e.name]
    q.qdit_destroy(ctx)
    assert len(names) == 1 and kernel + "<" in names[0], names
