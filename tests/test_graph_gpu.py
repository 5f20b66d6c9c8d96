"""kv_store + kv_load captured into a CUDA graph and replayed.

The calls order their side-stream work with an event on the caller's stream
and a join back to it, which stream capture turns into graph edges; the
zero-copy mode allocates nothing per call.  A captured store/restore is
replayed twice with new KV written between the replays and each replay is
checked against the oracle.
"""
import os
import subprocess
import sys
import time

import numpy as np
import pytest
import torch

import oracle
from gpu_util import POISON, device_pool, first_mismatch, host_layers, kvx, np_of, oracle_load, oracle_store, pinned_chunks
from paper_2609_15021_gb300 import synth

pytestmark = pytest.mark.gpu


def test_store_restore_replayed_from_a_cuda_graph(orc):
    k = kvx()
    spec = oracle.PoolSpec(4, 64, 16, 8, 128, 2, oracle.HND)
    C, n_used = 256, 40
    T = n_used * 16 - 7
    src = device_pool(spec, host_layers(spec, 1))
    dst = device_pool(spec)
    ta = synth.permuted_table(64, n_used, 2)
    tb = synth.permuted_table(64, n_used, 3)
    ta_d, tb_d = torch.from_numpy(ta).cuda(), torch.from_numpy(tb).cuda()
    host = pinned_chunks(orc, spec, 0, T, C)
    ctx = k.kv_ctx_create(0)
    torch.cuda.synchronize()  # the poisoned pool was filled on the default stream
    try:
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):  # warm up outside the capture
            k.kv_store(ctx, src, ta_d, 0, T, C, host)
            k.kv_load(ctx, dst, tb_d, 0, T, C, host)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s, capture_error_mode="thread_local"):
            k.kv_store(ctx, src, ta_d, 0, T, C, host)
            k.kv_load(ctx, dst, tb_d, 0, T, C, host)
        for seed in (10, 11):
            new = host_layers(spec, seed)
            for l, a in enumerate(new):
                src.layers[l].copy_(torch.from_numpy(a))
            for t in dst.layers:
                t.fill_(POISON)
            torch.cuda.synchronize()
            g.replay()
            torch.cuda.synchronize()
            want, _ = oracle_store(orc, spec, new, ta, 0, T, C)
            for h, w in zip(host, want):
                assert first_mismatch(np_of(h), w) is None, seed
            loaded, _ = oracle_load(orc, spec, [np.full(spec.layer_bytes, POISON, np.uint8)] * 4, tb, 0, T, C, want)
            for l in range(4):
                assert first_mismatch(np_of(dst.layers[l]), loaded[l]) is None, (seed, l)
        assert k.kv_get_device_error(ctx) == -1
    finally:
        k.kv_ctx_destroy(ctx)


def test_tier_calls_during_a_capture(orc):
    """Tier calls keep host bookkeeping, so one given a capturing stream is
    refused (KVX_EINVAL) and the capture goes on; calls without a stream
    (reserve, lookups) made while the thread captures leave the capture alone.
    The captured store is replayed, then committed outside the capture, and
    its bytes match the oracle."""
    k = kvx()
    spec = oracle.PoolSpec(4, 64, 16, 8, 128, 2, oracle.HND)
    C, n_used = 256, 32
    T = n_used * 16
    layers_np = host_layers(spec, 5)
    src = device_pool(spec, layers_np)
    ta = synth.permuted_table(64, n_used, 6)
    ta_d = torch.from_numpy(ta).cuda()
    keys = [901, 902]
    tier = k.KvTier(orc.chunk_bytes(spec, C), 4, shared_name=f"/kvx_graph_{__import__('os').getpid()}", create=True)
    ctx = k.kv_ctx_create(0)
    try:
        s = torch.cuda.Stream()
        slots = tier.reserve_many(keys)
        with torch.cuda.stream(s):  # warm up outside the capture
            k.kv_store(ctx, src, ta_d, 0, T, C, slots)
        s.synchronize()
        tier.reserve(903)                       # an entry with GPU work pending when the capture starts
        tier.commit(903, stream=s)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):     # the strictest capture mode: global
            k.kv_store(ctx, src, ta_d, 0, T, C, slots)
            for call in (lambda: tier.commit_many(keys, stream=s), lambda: tier.acquire(903, stream=s),
                         lambda: tier.release(903, stream=s)):
                with pytest.raises(k.KvxError) as e:
                    call()
                assert e.value.status == k.KVX_EINVAL
            assert tier.prefix_hits(keys) == 0  # host-side calls go on (with event queries) inside the capture
            tier.reserve(904)
        g.replay()
        tier.commit_many(keys, stream=s)
        s.synchronize()
        assert tier.prefix_hits(keys) == 2
        want, _ = oracle_store(orc, spec, layers_np, ta, 0, T, C)
        for c, key in enumerate(keys):
            got = tier.acquire(key, k.KVX_NO_STREAM)
            assert first_mismatch(np_of(got), want[c]) is None, c
            tier.release(key, k.KVX_NO_STREAM)
        assert k.kv_get_device_error(ctx) == -1
    finally:
        k.kv_ctx_destroy(ctx)
        tier.close()


def test_first_calls_of_a_context_inside_a_capture(orc):
    """A context's first transfer, or its first after more than 1 s, is when the
    library reads the chunks' host pages behind a host function on the stream.
    Made on a capturing stream, that read is skipped: nothing of it enters the
    graph (a replayed host function would wait on a job that no longer exists).
    The capture below is the new context's very first call, and a second one
    follows 1.1 s later; both graphs replay twice bit-exactly."""
    import time
    k = kvx()
    spec = oracle.PoolSpec(4, 64, 16, 8, 128, 2, oracle.HND)
    C, n_used = 256, 40
    T = n_used * 16 - 7
    src = device_pool(spec, host_layers(spec, 21))
    dst = device_pool(spec)
    ta = synth.permuted_table(64, n_used, 22)
    tb = synth.permuted_table(64, n_used, 23)
    ta_d, tb_d = torch.from_numpy(ta).cuda(), torch.from_numpy(tb).cuda()
    host = pinned_chunks(orc, spec, 0, T, C)
    ctx = k.kv_ctx_create(0)
    try:
        s = torch.cuda.Stream()
        torch.cuda.synchronize()
        graphs = []
        for pause in (0.0, 1.1):
            time.sleep(pause)
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):   # global capture mode
                k.kv_store(ctx, src, ta_d, 0, T, C, host)
                k.kv_load(ctx, dst, tb_d, 0, T, C, host)
            graphs.append(g)
        for i, g in enumerate(graphs * 2):
            new = host_layers(spec, 30 + i)
            for l, a in enumerate(new):
                src.layers[l].copy_(torch.from_numpy(a))
            for t in dst.layers:
                t.fill_(POISON)
            torch.cuda.synchronize()
            g.replay()
            torch.cuda.synchronize()
            want, _ = oracle_store(orc, spec, new, ta, 0, T, C)
            for h, w in zip(host, want):
                assert first_mismatch(np_of(h), w) is None, i
            loaded, _ = oracle_load(orc, spec, [np.full(spec.layer_bytes, POISON, np.uint8)] * 4, tb, 0, T, C, want)
            for l in range(4):
                assert first_mismatch(np_of(dst.layers[l]), loaded[l]) is None, (i, l)
        assert k.kv_get_device_error(ctx) == -1
    finally:
        k.kv_ctx_destroy(ctx)


def _first_device_moves_body():
    k = kvx()
    orc = oracle.c_oracle()
    spec = oracle.PoolSpec(2, 40, 16, 3, 40, 2, oracle.HND)  # page halves of 3,840 B: loads and stores
    C, T = 64, 37 * 16 - 5
    src_np, table = host_layers(spec, 51), synth.permuted_table(40, 37, 52)
    src, dst, tab = device_pool(spec, src_np), device_pool(spec), torch.from_numpy(table).cuda()
    want, _ = oracle_store(orc, spec, src_np, table, 0, T, C)
    dev = [torch.full((w.size,), POISON, dtype=torch.uint8, device="cuda") for w in want]
    ctx = k.kv_ctx_create(0)
    s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    spin = torch.cuda.Stream()
    with torch.cuda.graph(g, stream=s):  # global capture mode
        with torch.cuda.stream(spin):
            torch.cuda._sleep(2_000_000_000)  # a second of other work on the GPU, outside the capture
        t = time.perf_counter()
        k.kv_pack(ctx, src, tab, 0, T, C, dev, stream=s)
        k.kv_unpack(ctx, dst, tab, 0, T, C, dev, stream=s)
        t = time.perf_counter() - t
    assert t < 0.3, f"the first calls took {t:.2f} s: they waited for the GPU"
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()
    loaded, _ = oracle_load(orc, spec, [np.full(spec.layer_bytes, POISON, np.uint8)] * 2, table, 0, T, C, want)
    for d, w in zip(dev, want):
        assert first_mismatch(np_of(d), w) is None
    for t, w in zip(dst.layers, loaded):
        assert first_mismatch(np_of(t), w) is None
    assert k.kv_get_device_error(ctx) == -1
    k.kv_ctx_destroy(ctx)
    print("FIRST_MOVES_OK")


def test_first_device_moves_of_a_process_inside_a_capture():
    """The context's set-up loads every load/store kernel: a process's first kv_pack and kv_unpack,
    here in a capture beside other work, load nothing and wait for nothing."""
    here = os.path.dirname(os.path.abspath(__file__))
    code = (f"import sys; sys.path[:0] = [{here!r}, {os.path.dirname(here)!r}]; "
            "import test_graph_gpu as t; t._first_device_moves_body()")
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300, cwd=here)
    assert r.returncode == 0 and "FIRST_MOVES_OK" in r.stdout, r.stdout[-3000:] + r.stderr[-3000:]
