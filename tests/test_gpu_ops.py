"""GPU parity of the kernel-level projection op (uad_linear) against an fp64 reference of the
same bf16 operands (tolerance: fp32 accumulation, 1e-5 of the output scale)."""
import numpy as np
import pytest
import torch

import paper_2609_37772_gb300 as uad
from uad_inputs import round_to_bf16

pytestmark = pytest.mark.gpu


def run_linear(x, w, bias, fn=None):
    fn = fn or uad.uad_linear
    M, K = x.shape
    N = w.shape[1]
    xd = torch.from_numpy(round_to_bf16(x)).to(torch.bfloat16).cuda()
    wd = torch.from_numpy(uad.tile_weight(w).view(np.int16)).cuda()
    bd = None if bias is None else torch.from_numpy(bias).cuda()
    out = torch.full((M, N), float("nan"), device="cuda")
    rc = fn(xd.data_ptr(), wd.data_ptr(), None if bd is None else bd.data_ptr(), out.data_ptr(), M, N, K,
            torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return rc, out.cpu().numpy()


def reference(x, w, bias):
    r = round_to_bf16(x).astype(np.float64) @ round_to_bf16(w).astype(np.float64)
    return r + (0 if bias is None else bias.astype(np.float64))


@pytest.mark.parametrize("M,N,K", [(50, 1024, 2048), (50, 2560, 1024), (64, 8192, 1024), (1, 128, 64),
                                   (130, 384, 4096), (50, 1024, 4096)])
def test_linear_matches_reference(M, N, K):
    rng = np.random.default_rng(M * 7 + N + K)
    x = rng.normal(size=(M, K)).astype(np.float32)
    w = (rng.normal(size=(K, N)) * 0.02).astype(np.float32)
    bias = rng.normal(size=N).astype(np.float32)
    rc, out = run_linear(x, w, bias)
    assert rc == 0
    ref = reference(x, w, bias)
    assert np.abs(out - ref).max() <= 1e-5 * np.abs(ref).max()


# Shapes that take the persistent wide form on a 152-SM GB300, with each of its tile widths and
# ragged last token tiles (plan of the busiest CTA's work):
#   (2560, 2048, 64): 16 weight tiles x 14 tiles of 192 tokens (the last 64)
#   (3000, 1024, 128): 8 x 16 tiles of 192 tokens (the last 120)
#   (2400, 1024, 128): 8 x 19 tiles of 128 tokens (the last 96)
#   (800, 2560, 192): 20 x 7 tiles of 128 tokens (the last 32)
@pytest.mark.parametrize("M,N,K", [(2560, 2048, 64), (3000, 1024, 128), (2400, 1024, 128), (800, 2560, 192)])
def test_linear_wide_tiles_match_reference(M, N, K):
    rng = np.random.default_rng(M + N + K)
    x = rng.normal(size=(M, K)).astype(np.float32)
    w = (rng.normal(size=(K, N)) * 0.02).astype(np.float32)
    bias = rng.normal(size=N).astype(np.float32)
    rc, out = run_linear(x, w, bias)
    assert rc == 0
    ref = reference(x, w, bias)
    assert np.abs(out - ref).max() <= 1e-5 * np.abs(ref).max()


# The cluster form (K splits exchanged between CTAs) where a share is ragged or empty, and the long-K shapes
# of many rows that it takes over from the wide form:
#   (1, 128, 512): one token row for eight CTAs; (9, 256, 640): two rows each for five CTAs, ten k-blocks over eight;
#   (63, 128, 4096): seven CTAs with eight rows, one with seven; (65, 256, 1024): a second tile of one row;
#   (637, 1024, 2048), (1200, 512, 2112): two and three splits of ragged last tiles
# and tiles of 64 weight rows (33 to 64 tokens): (33, 128, 64): one k-block, no splits; (47, 384, 1600): an odd
# number of tokens, more k-blocks than slots; (64, 3200, 320): the widest N that they serve;
# boxes of 16 token rows, five slots walked more than once, and the first size past them: (16, 6400, 1088), (17, 128, 128)
@pytest.mark.parametrize("M,N,K", [(1, 128, 512), (9, 256, 640), (63, 128, 4096), (65, 256, 1024), (637, 1024, 2048),
                                   (1200, 512, 2112), (33, 128, 64), (47, 384, 1600), (64, 3200, 320),
                                   (16, 6400, 1088), (17, 128, 128)])
def test_linear_cluster_shares_match_reference(M, N, K):
    rng = np.random.default_rng(M + N + K)
    x = rng.normal(size=(M, K)).astype(np.float32)
    w = (rng.normal(size=(K, N)) * 0.02).astype(np.float32)
    rc, out = run_linear(x, w, None)
    assert rc == 0
    ref = reference(x, w, None)
    assert np.abs(out - ref).max() <= 1e-5 * np.abs(ref).max()


@pytest.mark.parametrize("M,N,K", [(16, 256, 512), (200, 8192, 128), (530, 2560, 128)])
def test_linear_takes_outputs_and_biases_at_any_float_address(M, N, K):
    """out and bias one float past a 16-byte boundary, on the cluster, narrow and wide forms: stores and
    loads fall back to single floats, and nothing around the output is written."""
    rng = np.random.default_rng(M + N + K)
    x = torch.from_numpy(rng.normal(size=(M, K)).astype(np.float32)).to(torch.bfloat16).cuda()
    w = (rng.normal(size=(K, N)) * 0.02).astype(np.float32)
    wd = torch.from_numpy(uad.tile_weight(w).view(np.int16)).cuda()
    room = torch.full((M * N + 8,), float("nan"), device="cuda")
    bias = torch.from_numpy(rng.normal(size=N + 1).astype(np.float32)).cuda()
    rc = uad.uad_linear(x.data_ptr(), wd.data_ptr(), bias[1:].data_ptr(), room[1:].data_ptr(), M, N, K,
                        torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert rc == 0
    got = room.cpu().numpy()
    ref = x.float().cpu().numpy().astype(np.float64) @ round_to_bf16(w).astype(np.float64) + bias[1:].cpu().numpy()
    assert np.abs(got[1:1 + M * N].reshape(M, N) - ref).max() <= 1e-5 * np.abs(ref).max()
    assert np.isnan(got[0]) and np.isnan(got[1 + M * N:]).all()


def test_linear_rejects_bad_shapes():
    assert uad.uad_linear(1, 1, None, 1, 50, 100, 64, None) == uad.UAD_EINVAL
    assert uad.uad_linear(1, 1, None, 1, 0, 128, 64, None) == uad.UAD_EINVAL
    assert uad.uad_linear(None, 1, None, 1, 50, 128, 64, None) == uad.UAD_EINVAL


@pytest.mark.parametrize("M,N,K", [(16, 512, 1536), (50, 1024, 512), (160, 8192, 128), (637, 1024, 2048)])
def test_linear_reads_weights_and_bias_in_stream_order(M, N, K):
    """A call's bias is the output of the call just before it on the stream, its weights are copied there in
    between: on the cluster form (16 and 50 rows, long K) and the narrow form, each sees them complete."""
    rng = np.random.default_rng(M + N + K)
    st = torch.cuda.Stream()
    big = 3072   # rows of the call that computes the bias: long enough that the next call's CTAs could start beside it
    xb = torch.from_numpy(rng.normal(size=(big, K)).astype(np.float32)).to(torch.bfloat16).cuda()
    x = torch.from_numpy(rng.normal(size=(M, K)).astype(np.float32)).to(torch.bfloat16).cuda()
    ws = [(rng.normal(size=(K, N)) * 0.02).astype(np.float32) for _ in range(3)]
    tiled = [torch.from_numpy(uad.tile_weight(w).view(np.int16)).cuda() for w in ws]
    refs = [x.float().cpu().numpy().astype(np.float64) @ round_to_bf16(w).astype(np.float64) for w in ws]
    lasts = [xb[-1].float().cpu().numpy().astype(np.float64) @ round_to_bf16(w).astype(np.float64) for w in ws]
    wt = torch.zeros_like(tiled[0])
    outb = torch.zeros(big, N, device="cuda")
    outs = [torch.zeros(M, N, device="cuda") for _ in range(12)]
    torch.cuda.synchronize()
    for i, out in enumerate(outs):
        assert uad.uad_linear(xb.data_ptr(), tiled[i % 3].data_ptr(), None, outb.data_ptr(), big, N, K, st.cuda_stream) == 0
        if i % 2:   # with the weights' copy between the two calls, and without
            with torch.cuda.stream(st):
                wt.copy_(tiled[(i + 1) % 3])
        w = wt if i % 2 else tiled[(i + 1) % 3]
        assert uad.uad_linear(x.data_ptr(), w.data_ptr(), outb[-1].data_ptr(), out.data_ptr(), M, N, K, st.cuda_stream) == 0
    torch.cuda.synchronize()
    for i, out in enumerate(outs):
        want = refs[(i + 1) % 3] + lasts[i % 3]
        assert np.abs(out.cpu().numpy() - want).max() <= 1e-5 * np.abs(want).max(), i


@pytest.mark.parametrize("M,N,K", [(16, 4608, 1536), (16, 6144, 1536), (16, 1536, 6144), (1, 1024, 6144), (32, 1536, 6144),
                                   (50, 1024, 4096), (64, 512, 4096), (64, 1536, 6144), (100, 1024, 4096), (13, 384, 8192)])
def test_linear_sums_few_rows_in_short_runs(M, N, K):
    """The tensor cores' accumulation truncates: each step of 16 products loses up to an ulp of the sum so far, half
    of one on average. Over positive products, where the sum grows evenly, a run of 256 so loses at most
    16 / 2 steps x 2^-24 = 4.8e-7 of it on average, and a longer run more."""
    g = torch.Generator(device="cuda")
    g.manual_seed(M + N + K)
    x = torch.randn((M, K), generator=g, device="cuda").abs().bfloat16()
    w = torch.randn((K, N), generator=g, device="cuda").mul_(0.02).abs().bfloat16()
    tiled = torch.from_numpy(uad.tile_weight(w.float().cpu().numpy()).view(np.int16)).cuda()
    out = torch.empty((M, N), device="cuda")
    assert uad.uad_linear(x.data_ptr(), tiled.data_ptr(), None, out.data_ptr(), M, N, K, torch.cuda.current_stream().cuda_stream) == 0
    ref = x.double() @ w.double()
    mean = ((out.double() - ref) / ref).mean().abs().item()
    print(f"{M} x {K} x {N}: mean relative error {mean:.2e}")
    assert mean <= 8 * 2.0 ** -24
