"""The persistent evaluation kernel's bounded waits, made to run out without any GPU fault: the
first completion count of every evaluation is told to wait for one arrival more than the kernel
ever makes, with a 1 ms limit. Every wait gives up, records its code and lets the launch wind
down; uad_finish reports the error; the same context then runs a correct chunk."""
import numpy as np
import pytest
import torch

import paper_2609_37772_gb300 as uad
from oracle.model import build_model
from oracle.uad import denoise
from uad_inputs import ARCHS, group_budgets, make_noise, make_prefix_kv, make_weights

pytestmark = pytest.mark.gpu


def test_expired_wait_is_reported_and_the_context_recovers():
    a = ARCHS["pi0_small"]
    blob = make_weights(a, seed=21)
    kv = make_prefix_kv(a, seed=21)
    noise = make_noise(a, seed=21)
    bud = group_budgets(a.chunk_len, [(0, 9, 3), (10, a.chunk_len - 1, 6)])
    ex = uad.Expert(a, blob)
    try:
        ex.set_prefix(0, *kv)
        names = {r["name"] for r in ex.profile(noise, bud[None])}
        assert names == {"begin", "step_kernel"}, names   # the persistent kernel serves this chunk
        ex.set_wait_limit(wait_ns=1_000_000, unreachable=1)
        ex.denoise(noise, bud[None])
        r = ex.finish(timeout_us=60_000_000, check=False)
        assert r["rc"] == uad.UAD_ECUDA, r["rc"]
        # whichever bounded wait ran out first recorded its code (51: a completion count; the
        # issuer's operand wait, 42, can expire first with a 1 ms limit)
        msg = uad.uad_last_error(ex.h).decode()
        assert "timed out (code" in msg, msg
        # released actions were never flagged: nothing reached the controller
        rc, _, ready, _ = ex.poll(0, min_ready=1, timeout_us=0)
        assert rc in (uad.UAD_ETIMEDOUT, uad.UAD_ESTATE) or not ready.any()
        ex.set_wait_limit()   # back to the 2 s default, counts reachable again
        ex.denoise(noise, bud[None])
        ok = ex.finish(timeout_us=60_000_000)
        ref = denoise(build_model(a, blob, kv).velocity, noise[0], bud)
        err = np.abs(ok["final"][0] - ref["final"]).max() / np.abs(ref["final"]).max()
        print(f"after recovery: max rel err {err:.2e}")
        assert ok["rc"] == 0 and err <= 2e-2 and ok["evals"] == 6
    finally:
        ex.close()


def test_expired_wait_falls_back_to_per_operation_kernels():
    """After a wait of the persistent kernel ran out (as it would if its CTAs were not all
    resident), the context runs later chunks on the per-operation kernels, correctly, until the
    wait limit is set again."""
    a = ARCHS["pi0_small"]
    blob = make_weights(a, seed=22)
    kv = make_prefix_kv(a, seed=22)
    noise = make_noise(a, seed=22)
    bud = group_budgets(a.chunk_len, [(0, 9, 3), (10, a.chunk_len - 1, 6)])
    ex = uad.Expert(a, blob)
    try:
        ex.set_prefix(0, *kv)
        ex.set_wait_limit(wait_ns=1_000_000, unreachable=1)
        ex.denoise(noise, bud[None])
        r = ex.finish(timeout_us=60_000_000, check=False)
        assert r["rc"] == uad.UAD_ECUDA, r["rc"]
        msg = uad.uad_last_error(ex.h).decode()
        assert "per-operation kernels" in msg, msg
        names = {r["name"] for r in ex.profile(noise, bud[None])}
        assert "step_kernel" not in names and "qkv_proj" in names, names
        ex.denoise(noise, bud[None])
        ok = ex.finish(timeout_us=60_000_000)
        ref = denoise(build_model(a, blob, kv).velocity, noise[0], bud)
        err = np.abs(ok["final"][0] - ref["final"]).max() / np.abs(ref["final"]).max()
        print(f"per-operation fall-back: max rel err {err:.2e}")
        assert ok["rc"] == 0 and err <= 2e-2 and ok["evals"] == 6
        ex.set_wait_limit()
        names = {r["name"] for r in ex.profile(noise, bud[None])}
        assert names == {"begin", "step_kernel"}, names
    finally:
        ex.close()


def test_a_cached_chunk_runs_once_after_a_wait_ran_out():
    """Four robots of 16 tokens leave the persistent kernel no room for their flow times, so their chunks run on
    the per-operation kernels beside one-robot chunks on the persistent one. Their cached graph keeps its
    own number of steps when a wait of the persistent kernel runs out later: the chunk takes as long as
    before (not twice) and gives the same bits."""
    a = ARCHS["pi0_small"].replace(name="pi0_small_h16", chunk_len=16)
    ex = uad.Expert(a, make_weights(a, seed=23), max_batch=4)
    noise = make_noise(a, batch=4, seed=23)
    bud = np.stack([group_budgets(16, [(0, 3, 4 + b), (4, 15, 16)]) for b in range(4)])
    dev = torch.from_numpy(noise).cuda()
    stream = torch.cuda.Stream()

    def chunk():
        ms = []
        for _ in range(6):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record(stream)
            ex.denoise(dev, bud, stream=stream)
            t1.record(stream)
            r = ex.finish(timeout_us=60_000_000)
            torch.cuda.synchronize()
            ms.append(t0.elapsed_time(t1))
        return r, min(ms)

    try:
        for b in range(4):
            ex.set_prefix(b, *make_prefix_kv(a, robot=b, seed=23))
        names = {r["name"] for r in ex.profile(noise, bud)}
        assert "step_kernel" not in names, names
        ex.set_wait_limit(wait_ns=1_000_000, unreachable=1)
        first, t_first = chunk()
        ex.denoise(noise[:1], bud[:1])
        r = ex.finish(timeout_us=60_000_000, check=False)
        assert r["rc"] == uad.UAD_ECUDA and "per-operation kernels" in uad.uad_last_error(ex.h).decode()
        again, t_again = chunk()
        print(f"16 steps of four robots: {t_first:.3f} ms, after the expired wait {t_again:.3f} ms")
        assert np.array_equal(again["final"], first["final"]) and again["evals"] == first["evals"] == 16
        assert t_again <= 1.4 * t_first
    finally:
        ex.close()


@pytest.mark.parametrize("M,N,K", [(16, 512, 6144), (50, 1024, 4096), (160, 8192, 512), (600, 4096, 1024), (2, 1536, 6144)])
def test_a_stopped_projection_harms_no_other_call(M, N, K):
    """A projection that runs as if one of its waits had run out (cluster form with 128 and 64 weight rows, narrow
    and persistent form): it ends at once, uad_linear_status reports it once, and the calls after it on
    its stream and beside it on another give what they always give, 1500 of them, so that each error word
    is used again."""
    rng = np.random.default_rng(M + N + K)
    x = torch.from_numpy(rng.normal(size=(M, K)).astype(np.float32)).to(torch.bfloat16).cuda()
    w = torch.from_numpy(uad.tile_weight((rng.normal(size=(K, N)) * 0.02).astype(np.float32)).view(np.int16)).cuda()
    s0, s1 = torch.cuda.Stream(), torch.cuda.Stream()
    outs = [torch.full((M, N), float("nan"), device="cuda") for _ in range(12)]
    torch.cuda.synchronize()

    def call(entry, out, s):
        assert entry(x.data_ptr(), w.data_ptr(), None, out.data_ptr(), M, N, K, s.cuda_stream) == 0

    uad.uad_linear_status()
    call(uad.uad_linear, outs[0], s0)
    torch.cuda.synchronize()
    assert uad.uad_linear_status() == uad.UAD_OK
    for _ in range(5):
        call(uad.uad_linear_check, outs[1], s0)
        call(uad.uad_linear, outs[2], s1)
        call(uad.uad_linear, outs[3], s0)
    torch.cuda.synchronize()
    assert uad.uad_linear_status() == uad.UAD_ECUDA
    assert uad.uad_linear_status() == uad.UAD_OK
    call(uad.uad_linear_check, outs[1], s0)
    for i in range(1500):
        call(uad.uad_linear, outs[4 + i % 8], s0 if i % 3 else s1)
    torch.cuda.synchronize()
    assert torch.isfinite(outs[0]).all()
    assert all(torch.equal(o, outs[0]) for o in outs[2:])
