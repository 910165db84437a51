"""Inputs at the edges of what the entry points take: they are answered, or reported, and touch nothing else."""
import threading
import time

import numpy as np
import pytest
import torch

import oracle
from paper_2605_08692_b200 import binding, build, synth
from test_gpu_parity import DEV, INT4, NVFP4, dev_bf16, host, layer, table_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def fit_only(W, mode, I, rounds, init, ws):
    """aaac_fit_layer on device tensors; returns the tables and the status bits."""
    N, K = W.shape
    g = binding.group_of(mode)
    T01 = torch.zeros(2, 16, dtype=torch.float32, device=DEV)
    scales = torch.zeros(N, K // g, dtype=torch.int16 if mode == INT4 else torch.uint8, device=DEV)
    ts, st = torch.ones(1, dtype=torch.float32, device=DEV), torch.zeros(1, dtype=torch.int32, device=DEV)
    binding.fit_layer(W, mode, I=I, n_outer=rounds, init=init, T01=T01, scales=scales, tensor_scale=ts, ws=ws, dev_status=st)
    torch.cuda.synchronize()
    return host(T01), int(st.item())


def test_quantile_start_with_nan_groups_stays_inside_its_workspace():
    """A NaN gives its INT4 group the smallest scale, 2^-126, so the group's other weights become w 2^126: far outside the
    histogram's range, and 4096 times them outside FP32's.  Every weight has to be collected from the bin it was counted in
    all the same -- here 1.6 million of them, six times what the candidate list holds."""
    N, K = 4096, 1024
    rng = np.random.default_rng(3)
    w = (0.02 * rng.standard_normal((N, K // 128, 128))).astype(np.float32)
    bad = rng.random((N, K // 128)) < 0.4
    w[bad] = rng.uniform(9.8e-4, 3.9e-3, (int(bad.sum()), 128)).astype(np.float32)
    W = synth.f32_to_bf16_bits(w.reshape(N, K)).reshape(N, K // 128, 128)
    W[bad, 17] = 0x7FC0
    first = np.argwhere(bad)[0]
    W[first[0], first[1], 40] = 0x4080                     # 4: infinite once normalised
    size, guard = binding.workspace_bytes(INT4, N, K), 16 << 20
    buf = torch.full((size + guard,), 0xA5, dtype=torch.uint8, device=DEV)
    _, status = fit_only(dev_bf16(W.reshape(N, K)), INT4, torch.ones(K, device=DEV), 0, binding.INIT_QUANTILE, buf[:size])
    assert status & binding.DEV_NONFINITE
    assert bool((buf[size:] == 0xA5).all())


def host_call(W, X, mode, rounds, init=binding.INIT_QUANTILE, pinned=True, queue_only=False):
    """A host-buffer call with all its buffers: a function that makes it, and the outputs it fills."""
    N, K, T = W.shape[0], W.shape[1], X.shape[0]
    pin = lambda t: t.pin_memory() if pinned else t
    out = dict(T01_host=torch.empty(2, 16), T01_bf16_host=torch.empty(2, 16, dtype=torch.int16),
               scales_host=torch.empty(N, K // binding.group_of(mode), dtype=torch.int16 if mode == INT4 else torch.uint8),
               tensor_scale_host=torch.empty(1), codes_host=torch.empty(N, K // 2, dtype=torch.uint8),
               err_out_host=torch.empty(2, dtype=torch.float64))
    out = {k: pin(v) for k, v in out.items()}
    Wh, Xh = pin(torch.from_numpy(W.view(np.int16))), pin(torch.from_numpy(X.view(np.int16)))
    ws = torch.empty(binding.host_workspace_bytes(mode, N, K, T), dtype=torch.uint8, device=DEV)
    if queue_only:
        st = pin(torch.zeros(1, dtype=torch.int32))
        return lambda: binding.quantize_layer_host_async(Wh, Xh, mode, n_outer=rounds, init=init, ws=ws, status_host=st, **out), out
    return lambda: binding.quantize_layer_host(Wh, Xh, mode, n_outer=rounds, init=init, ws=ws, **out), out


# (4096 x 1024 and 4096 x 512: a quarter and a half of the blocks share the column slab of the infinite importance)
@pytest.mark.parametrize("mode,N,K", [(NVFP4, 4096, 1024), (NVFP4, 4096, 512), (INT4, 4096, 1024), (INT4, 64, 256)])
@pytest.mark.parametrize("value", [0x7F80, 0xFF80, 0x7FC0])
def test_nonfinite_activations_are_reported_as_such(mode, N, K, value):
    """An infinite or NaN importance makes a cell's sums infinite: the blocks' exchange of sums has to end all the same."""
    W, X = layer(mode, N, K, name=f"infact/{mode}/{N}x{K}")
    X[5, 33] = value
    r = binding.quantize_layer(dev_bf16(W), mode, X=dev_bf16(X), n_outer=5, init=binding.INIT_QUANTILE, want_trace=True)
    torch.cuda.synchronize()
    assert int(r["status"].item()) == binding.DEV_NONFINITE
    with pytest.raises(binding.AaacError, match="Inf or NaN"):
        host_call(W, X, mode, 5)[0]()


@pytest.mark.parametrize("mode", [INT4, NVFP4])
@pytest.mark.parametrize("n_inner", [1, 3])
def test_nonfinite_weights_are_reported_after_rounds(mode, n_inner):
    W, X = layer(mode, 300, 768, name=f"infw/{mode}")
    W[7, 100], W[200, 5], W[31, 700] = 0x7F80, 0x7FC0, 0xFF80
    r = binding.quantize_layer(dev_bf16(W), mode, X=dev_bf16(X), n_outer=3, n_inner=n_inner, init=binding.INIT_QUANTILE, want_trace=True)
    torch.cuda.synchronize()
    assert int(r["status"].item()) & (binding.DEV_NONFINITE | binding.DEV_TIMEOUT) == binding.DEV_NONFINITE


@pytest.mark.parametrize("far", [30.0, 1000.0])
def test_user_tables_far_outside_the_weights(far):
    """Every weight is `far` and more away from its entry, and one block holds the whole layer: the first objective is the
    largest sum a pass can have."""
    W, X = layer(INT4, 16, 256, name="fartables")
    T0 = np.stack([far + np.arange(16), far + 8 + np.arange(16)]).astype(np.float32)
    o = oracle.fit_layer(W, INT4, 128, 2, X=X, init="user", T_init=T0)
    r = binding.quantize_layer(dev_bf16(W), INT4, X=dev_bf16(X), n_outer=2, init=binding.INIT_USER, T01_init=torch.from_numpy(T0).to(DEV),
                               want_trace=True)
    torch.cuda.synchronize()
    assert int(r["status"].item()) == 0
    assert np.allclose(host(r["trace"]), o["trace"], rtol=1e-4)
    assert table_close(host(r["T01"]), o["T"])[0]


def test_an_entry_of_one_weight_of_hardly_any_importance_moves():
    """The sums over blocks are integers: their step has to lie far below every cell's weight, here 2^-60 of a channel's."""
    N, K = 16, 256
    rng = np.random.default_rng(8)
    w = rng.uniform(-0.07, 0.07, (N, K)).astype(np.float32)
    w[:, ::128] = -0.1                               # every group's largest magnitude, on the negative side ...
    w[0, 0] = 0.1                                    # ... but one: the only weight next to the uppermost entries
    I = np.ones(K, np.float32)
    I[0] = 2.0 ** -60
    T0 = np.stack([np.append(np.linspace(-7, 5, 15), 6.6), np.append(np.linspace(-6.5, 5.2, 15), 6.7)]).astype(np.float32)
    W = synth.f32_to_bf16_bits(w)
    o = oracle.fit_layer(W, INT4, 128, 1, I=I, init="user", T_init=T0)
    assert (np.abs(o["T"][:, 15] - T0[:, 15]) > 0.2).sum() == 1
    r = binding.quantize_layer(dev_bf16(W), INT4, I=torch.from_numpy(I).to(DEV), n_outer=1, init=binding.INIT_USER,
                               T01_init=torch.from_numpy(T0).to(DEV))
    torch.cuda.synchronize()
    assert table_close(host(r["T01"]), o["T"])[0]


@pytest.mark.parametrize("mode,N,K", [(INT4, 64, 512), (NVFP4, 200, 640)])
def test_negative_importances_of_the_callers(mode, N, K):
    """Importances are sums of squares, but nothing checks a caller's: a few negative ones give finite, if odd, sums."""
    g = binding.group_of(mode)
    W, X = layer(mode, N, K, name=f"neg/{mode}")
    I = oracle.act_stats(X)
    I[5::97] *= -0.25
    o = oracle.fit_layer(W, mode, g, 1, I=I, init="grid")
    r = binding.quantize_layer(dev_bf16(W), mode, I=torch.from_numpy(I).to(DEV), n_outer=1, init=binding.INIT_GRID)
    torch.cuda.synchronize()
    assert table_close(host(r["T01"]), o["T"], rel=1e-4)[0]      # (terms of both signs cancel: ten times the usual bar)


@pytest.mark.parametrize("mode", [INT4, NVFP4])
def test_quantile_start_with_room_for_some_of_the_bins(mode):
    """Which bins get space in a list that cannot hold all of them goes by the requests' slots, which every lane of a warp
    writes and one reads.  Bins of one value each are answered with or without space: the tables are those of a list that
    holds everything, whatever fits."""
    N, K, g = 300, 768, binding.group_of(mode)
    rng = np.random.default_rng(6)
    vals = (np.arange(-20, 21) * 0.33).astype(np.float32)          # 41 values in as many bins, 2 to 11 thousand weights each
    p = np.exp(-0.5 * (np.arange(-20, 21) / 9.0) ** 2)
    w = rng.choice(vals, size=(N, K), p=p / p.sum())
    w[:, ::g] = 7.0                                                # one scale for all groups
    W = dev_bf16(synth.f32_to_bf16_bits(w))
    I = torch.ones(K, device=DEV)
    want, status = fit_only(W, mode, I, 0, binding.INIT_QUANTILE, binding.alloc_workspace(mode, N, K, full=True))
    assert status == 0
    try:
        for cap in (1000, 6000, 20000, 60000, 150000):
            binding.debug_quantile_cap(cap)
            got, status = fit_only(W, mode, I, 0, binding.INIT_QUANTILE, binding.alloc_workspace(mode, N, K))
            assert status == 0 and np.array_equal(got, want), cap
    finally:
        binding.debug_quantile_cap(0)


def test_quantile_start_of_a_group_with_an_infinite_weight():
    """The group's scale is infinite, its finite weights are 0 of it and the infinite one is NaN, which sorts last: the start
    tables are the order statistics of that."""
    N, K = 40, 512
    W, _ = layer(INT4, N, K, name="infgroup")
    W[3, 140] = 0x7F80
    zeroed = W.copy()
    zeroed[3, 128:256] = 0
    s, ts = oracle.scales(zeroed, INT4, 128)
    x = oracle.normalise(zeroed, INT4, 128, s, ts).reshape(N, K).astype(np.float64)
    x[3, 140] = np.inf
    x = np.sort(x.reshape(-1))
    q = np.concatenate([np.arange(16) / 15.0, 1 / 30.0 + (1 - 1 / 30.0) * np.arange(16) / 15.0])
    pos = q * (x.size - 1)
    lo = np.floor(pos).astype(int)
    with np.errstate(invalid="ignore"):
        want = (x[lo] + (pos - lo) * (x[np.minimum(lo + 1, x.size - 1)] - x[lo])).astype(np.float32).reshape(2, 16)
    got, status = fit_only(dev_bf16(W), INT4, torch.ones(K, device=DEV), 0, binding.INIT_QUANTILE,
                           binding.alloc_workspace(INT4, N, K, full=True))
    assert status == binding.DEV_NONFINITE
    assert np.isfinite(want[:, :15]).all() and np.array_equal(got[:, :15], want[:, :15])
    assert not np.isfinite(got[:, 15]).any()


@pytest.mark.parametrize("T", [40, 1000])                   # one strip, and several
@pytest.mark.parametrize("value", [0x7F80, 0xFF80, 0x7FC0])
def test_importance_of_a_channel_with_a_nonfinite_activation(T, value):
    K = 264
    X = synth.activations(T, K, 4, f"nonfinite/{T}", kind="lognormal")
    want = oracle.act_stats(X)
    X[T // 2, 7] = value
    ws, I = binding.alloc_workspace(NVFP4, 1, K), torch.ones(K, dtype=torch.float32, device=DEV)
    for accumulate in (False, True):
        st = torch.zeros(1, dtype=torch.int32, device=DEV)
        binding.act_stats(dev_bf16(X), I, ws, accumulate=accumulate, dev_status=st)
        got = host(I)
        assert int(st.item()) == binding.DEV_NONFINITE and np.isnan(got[7])
        assert np.allclose(np.delete(got, 7), np.delete(want, 7) * (1 + accumulate), rtol=1e-6, atol=0)


def batch(mode, N, K, n):
    """n layers for quantize_layers"""
    g, out = binding.group_of(mode), []
    for l in range(n):
        W, X = layer(mode, N, K, name=f"batch/{mode}/{l}")
        out.append(dict(W=dev_bf16(W), X=dev_bf16(X), T01=torch.zeros(2, 16, device=DEV), T01_bf16=torch.zeros(2, 16, dtype=torch.bfloat16, device=DEV),
                        scales=torch.zeros(N, K // g, dtype=torch.int16 if mode == INT4 else torch.uint8, device=DEV),
                        tensor_scale=torch.ones(1, device=DEV), codes=torch.zeros(N, K // 2, dtype=torch.uint8, device=DEV),
                        ws=binding.alloc_workspace(mode, N, K, X.shape[0])))
    return out


def test_calls_of_other_threads_do_not_wait_for_a_host_buffer_call():
    """A host-buffer call returns when its stream is done, here behind about a second of other work; meanwhile another thread
    queues a batch, and runs a host-buffer call of its own."""
    W, X = layer(NVFP4, 1100, 2048, name="threads")
    layers, streams = batch(NVFP4, 256, 512, 2), [torch.cuda.Stream(), torch.cuda.Stream()]
    (call, mine), (slow_call, theirs) = host_call(W, X, NVFP4, 3), host_call(W, X, NVFP4, 3)
    run_batch = lambda: binding.quantize_layers(layers, NVFP4, n_outer=2, init=binding.INIT_QUANTILE)
    with torch.cuda.stream(streams[1]):                    # (what a first use loads or creates, every copy stream among it, is there)
        run_batch()
        for _ in range(8):
            call()
    with torch.cuda.stream(streams[0]):
        torch.cuda._sleep(1000)
        slow_call()
    want = {k: v.clone() for k, v in mine.items()}
    torch.cuda.synchronize()

    t0, at = time.perf_counter(), {}

    def behind_other_work():
        with torch.cuda.stream(streams[0]):
            torch.cuda._sleep(2_000_000_000)
            slow_call()
        at["slow call"] = time.perf_counter() - t0

    t = threading.Thread(target=behind_other_work)
    t.start()
    time.sleep(0.2)
    with torch.cuda.stream(streams[1]):
        run_batch()
        at["batch"] = time.perf_counter() - t0
        call()
        at["call"] = time.perf_counter() - t0
    t.join()
    torch.cuda.synchronize()
    assert at["call"] < 0.7 * at["slow call"], at
    for k, v in want.items():
        assert torch.equal(mine[k], v) and torch.equal(theirs[k], v), k


def test_pageable_host_buffers_give_what_page_locked_ones_do():
    W, X = layer(NVFP4, 1100, 2048, T=100, name="pageable")
    (pinned, want), (pageable, got) = host_call(W, X, NVFP4, 3), host_call(W, X, NVFP4, 3, pinned=False)
    pinned()
    before = binding.launch_count()
    pageable()
    assert binding.launch_count() - before == 9      # absmax, scales, plan, collect, select, importances (2), rounds, one pack of all rows
    for k in want:
        assert torch.equal(got[k], want[k]) or k == "err_out_host", k
    # (a lane adds up to 16 rows' terms in FP32, other rows where the pass runs by row ranges: 16 roundings of 2^-24)
    assert torch.allclose(got["err_out_host"], want["err_out_host"], rtol=1e-6)


def test_host_buffer_calls_beside_the_capture_of_one():
    """A captured call leaves nothing that other calls use in its graph: they go on while the capture is open, and the graph
    gives what the call gives."""
    W, X = layer(NVFP4, 1100, 2048, name="capture")
    (call, want), (captured, got) = host_call(W, X, NVFP4, 3, queue_only=True), host_call(W, X, NVFP4, 3, queue_only=True)
    beside, other = torch.cuda.Stream(), torch.cuda.Stream()
    captured()
    with torch.cuda.stream(beside):
        call()
    torch.cuda.synchronize()
    for t in got.values():
        t.zero_()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=other, capture_error_mode="relaxed"):
        captured()
        with torch.cuda.stream(beside):
            for _ in range(8):
                call()
    graph.replay()
    torch.cuda.synchronize()
    for k, v in want.items():
        assert torch.equal(got[k], v) or k == "err_out_host", k
    assert torch.allclose(got["err_out_host"], want["err_out_host"], rtol=1e-6)      # (row ranges, see above)


@pytest.mark.parametrize("mode,n_inner", [(INT4, 1), (NVFP4, 2)])
def test_captured_batch_gives_what_the_call_gives(mode, n_inner):
    """Side streams, the chain of dependent launches and the cooperative rounds as a graph."""
    layers = batch(mode, 300, 768, 3)
    run = lambda: binding.quantize_layers(layers, mode, n_outer=3, n_inner=n_inner, init=binding.INIT_QUANTILE)
    run()
    torch.cuda.synchronize()
    names = ("T01", "T01_bf16", "scales", "codes")
    want = [{k: d[k].clone() for k in names} for d in layers]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run()
    for d in layers:
        for k in names:
            d[k].zero_()
    for _ in range(2):
        graph.replay()
    torch.cuda.synchronize()
    for d, w in zip(layers, want):
        for k in names:
            assert torch.equal(d[k], w[k]), k


def test_prescaled_importances_may_replace_the_multipliers():
    N, K = 4096, 2048
    W, _ = layer(NVFP4, N, K, name="over_a")
    rng = np.random.default_rng(9)
    a, I = np.exp(0.5 * rng.standard_normal(K)).astype(np.float32), np.exp(rng.standard_normal(K)).astype(np.float32)
    Wd, a_then_I, Id = dev_bf16(W), torch.from_numpy(a).to(DEV), torch.from_numpy(I).to(DEV)
    want, I_want = torch.empty_like(Wd), torch.empty_like(Id)
    binding.prescale_columns(Wd, a_then_I, want, I=Id, I_out=I_want)
    got = torch.empty_like(Wd)
    binding.prescale_columns(Wd, a_then_I, got, I=Id, I_out=a_then_I)
    torch.cuda.synchronize()
    assert torch.equal(got, want) and torch.equal(a_then_I, I_want)
    assert np.array_equal(host(I_want), (I.astype(np.float64) / (a.astype(np.float64) ** 2)).astype(np.float32))
