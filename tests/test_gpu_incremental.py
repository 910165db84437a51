"""The incremental fit rounds, at sizes and on data where they can go wrong, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_08692_b200 import binding, build, synth
from test_gpu_parity import NVFP4, check_end_to_end_bits, dev_bf16, host, layer, run_fit_batch, table_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def check(W, X, rounds, init, name, inner=1, T01=None, place=dev_bf16):
    """Compares a fit with the oracle's (place: puts the weights on the device); returns the passes that were incremental, (first, end)."""
    o = oracle.fit_layer(W, NVFP4, 16, rounds, X=X, n_inner=inner, T_init=T01,
                         init={binding.INIT_QUANTILE: "quantile", binding.INIT_GRID: "grid", binding.INIT_USER: "user"}[init])
    ws = binding.alloc_workspace(NVFP4, W.shape[0], W.shape[1], X.shape[0])
    r = binding.quantize_layer(place(W), NVFP4, X=dev_bf16(X), n_outer=rounds, n_inner=inner, init=init, want_trace=True, ws=ws,
                               T01_init=None if T01 is None else torch.from_numpy(T01))
    torch.cuda.synchronize()
    assert int(r["status"].item()) == 0
    assert table_close(host(r["T01"]), o["T"])[0], name
    # (FP32 terms, 2^-24 each, and their sums over a lane's rows; where the entries meet every weight what is left is the
    # distance of the constants from the entries, 8 units in the last place at most: (2^-20 * 8)^2 of sum I)
    assert np.allclose(host(r["trace"])[:rounds], o["trace"], rtol=1e-5, atol=1e-10 * o["trace"][0]), name
    check_end_to_end_bits(r, o, name)
    return binding.debug_incremental(ws)


def rows_for(units, K):
    """Rows of a layer of K columns with so many units of 16 rows x 512 columns per block."""
    blocks = torch.cuda.get_device_properties(0).multi_processor_count
    return 16 * -(-units * blocks // -(-K // 512))


@pytest.mark.parametrize("K,units,extra,rounds,inner,init", [
    (512, 20, 0, 29, 1, binding.INIT_QUANTILE),         # one slab, the fewest units
    (512, 100, 16, 17, 1, binding.INIT_QUANTILE),       # few rounds
    (512, 24, -3, 27, 1, binding.INIT_QUANTILE),        # a last unit with rows missing
    (1008, 20, 5, 29, 1, binding.INIT_GRID),            # lanes without columns, ranges of units that differ by one; a start with equal entries
    (4096, 20, 16, 29, 1, binding.INIT_QUANTILE),       # short slabs
    (512, 6, -3, 3, 14, binding.INIT_QUANTILE),         # inner iterations
    (512, 7, 0, 1, 30, binding.INIT_QUANTILE),
    (1008, 11, 5, 2, 10, binding.INIT_QUANTILE),
])
def test_layers_of_few_units_per_block(K, units, extra, rounds, inner, init):
    W, X = layer(NVFP4, rows_for(units, K) + extra, K, T=64, name=f"incremental/{K}/{extra}")
    assert check(W, X, rounds, init, f"incremental {K} {units} {extra}", inner) == (3 if inner == 1 else 1, rounds * inner - 1)


def with_stride(ldw, offset):
    """Puts weights into a buffer of rows of ldw elements, the first one `offset` elements behind a 256-byte boundary."""
    def place(W):
        N, K = W.shape
        buf = torch.full((N * ldw + offset + 128,), float("nan"), dtype=torch.bfloat16, device="cuda")
        Wd = buf[offset:offset + N * ldw].view(N, ldw)[:, :K]
        Wd.copy_(dev_bf16(W))
        return Wd
    return place


@pytest.mark.parametrize("rounds,inner", [(29, 1), (3, 10)])
@pytest.mark.parametrize("ldw,offset,incremental", [(528, 0, True), (640, 16, True), (520, 0, False), (528, 8, False)])
def test_rows_apart_and_weights_off_32_bytes(ldw, offset, incremental, rounds, inner):
    """A piece is one 32-byte load: rows further apart than their width are taken, addresses that are not multiples of 32
    bytes are left to the full rounds."""
    W, X = layer(NVFP4, rows_for(20, 512) - 5, 512, T=64, name="incremental/stride")
    got = check(W, X, rounds, binding.INIT_QUANTILE, f"ldw {ldw} + {offset}", inner, place=with_stride(ldw, offset))
    assert got == ((3 if inner == 1 else 1, rounds * inner - 1) if incremental else (0, 0))


@pytest.mark.parametrize("rounds,inner", [(29, 1), (3, 10)])
def test_columns_without_importance(rounds, inner):
    """Whole groups of importance 0, undecided in every pass, and single columns of it."""
    W, X = layer(NVFP4, rows_for(20, 512), 512, T=64, name="incremental/zero")
    X[:, 64:192] = 0
    X[:, 200:512:7] = 0
    assert check(W, X, rounds, binding.INIT_QUANTILE, "zero importances", inner) == (3 if inner == 1 else 1, rounds * inner - 1)


@pytest.mark.parametrize("rounds,inner", [(29, 1), (3, 10)])
def test_wait_that_runs_out_is_reported(rounds, inner):
    """As of the full rounds: the status word says so, and the next fit with the workspace is what it was."""
    W, X = layer(NVFP4, rows_for(20, 512), 512, T=64, name="incremental/wait")
    Wd, Xd, ws = dev_bf16(W), dev_bf16(X), binding.alloc_workspace(NVFP4, *W.shape, X.shape[0])

    def fit():
        r = binding.quantize_layer(Wd, NVFP4, X=Xd, n_outer=rounds, n_inner=inner, init=binding.INIT_QUANTILE, ws=ws, want_trace=True)
        torch.cuda.synchronize()
        return r
    good = fit()
    assert int(good["status"].item()) == 0
    try:
        binding.debug_fit_wait(1, 1000)
        assert int(fit()["status"].item()) & binding.DEV_TIMEOUT and binding.debug_incremental(ws) == (0, 0)
    finally:
        binding.debug_fit_wait(0, 0)
    again = fit()
    assert int(again["status"].item()) == 0
    for k in ("T01", "codes", "scales", "trace", "err"):
        assert torch.equal(again[k], good[k]), k


def test_inner_iterations_from_equal_entries_are_not_tried():
    """The NVFP4 grid holds 0 twice: such a fit could not begin, and runs the launches of a small one."""
    W, X = layer(NVFP4, rows_for(8, 2048), 2048, T=64, name="incremental/2048/0")
    counts = []
    for rows in (64, len(W)):
        before = binding.launch_count()
        assert check(W[:rows].copy(), X, 3, binding.INIT_GRID, f"grid start, 3 x 10, {rows} rows", 10) == (0, 0)
        counts.append(binding.launch_count() - before)
    assert counts[0] == counts[1]


@pytest.mark.parametrize("units,rounds,inner,incremental", [
    (20, 25, 1, False), (20, 26, 1, True), (19, 40, 1, False), (40, 19, 1, False),
    (30, 2, 5, False), (30, 5, 4, False), (30, 1, 7, False), (14, 1, 10, False), (20, 1, 10, True), (7, 2, 10, False), (10, 2, 10, True), (8, 3, 7, False),
    (12, 3, 7, True), (16, 3, 5, True)])
def test_the_rule_takes_what_pays(units, rounds, inner, incremental):
    """(Layers may use some blocks fewer than there are, so that a block has a tenth more units.)"""
    W, X = layer(NVFP4, rows_for(units, 512), 512, T=64, name="incremental/rule")
    got = check(W, X, rounds, binding.INIT_QUANTILE, f"{units} units, {rounds} x {inner}", inner)
    assert got == ((3 if inner == 1 else 1, rounds * inner - 1) if incremental else (0, 0))


def tables(t0, t1):
    return np.stack([t0, t1]).astype(np.float32)


@pytest.mark.parametrize("start,rounds,inner", [
    ("far", 3, 10), ("far", 1, 30), ("apart", 29, 1), ("apart", 2, 14), ("twins", 3, 10)])
def test_fits_that_end_early_are_finished(start, rounds, inner):
    """Start tables beside the weights, whose entries jump: a cell's weight changes too much, or a breakpoint passes its
    neighbour, within the fit and within a round.  Equal entries: it cannot begin where it starts from the first pass."""
    N, K = rows_for(20, 512), 512
    W, X = layer(NVFP4, N, K, T=64, name="incremental/early")
    even = np.linspace(-6, 6, 16)
    T01 = {"far": tables(np.linspace(0.5, 1.5, 16), np.linspace(0.52, 1.52, 16)), "apart": tables(np.linspace(-6, -1, 16), np.linspace(1, 6, 16)),
           "twins": tables(np.where(np.arange(16) == 8, even[7], even), even)}[start]
    first, end = check(W, X, rounds, binding.INIT_USER, f"{start} {rounds} x {inner}", inner, T01)
    if start == "twins":
        assert (first, end) == (0, 0)
    else:
        assert first == (3 if inner == 1 else 1) and first < end < rounds * inner - 1


@pytest.mark.parametrize("rounds,inner", [(29, 1), (3, 10)])
@pytest.mark.parametrize("levels", [3, 17, 40])
def test_layers_of_few_distinct_weights(levels, rounds, inner):
    """Equal entries, empty cells and breakpoints that jump: the incremental rounds end early, or never begin."""
    N, K = rows_for(20, 512), 512
    W, X = layer(NVFP4, N, K, T=64, name=f"incremental/levels/{levels}")
    rng = np.random.default_rng(levels)
    values = np.sort(rng.standard_normal(levels)).astype(np.float32) * 0.02
    W = synth.f32_to_bf16_bits(values[rng.integers(0, levels, size=(N, K))])
    check(W, X, rounds, binding.INIT_GRID, f"levels {levels}", inner)


def followed(W, I, T, rounds):
    """The first pass behind the third at which a cell's weight falls below a quarter of the most it has had since, or the
    objective below a sixteenth of the most that it has been about the third round's tables, from a plain 64-bit run; the
    passes that can be incremental if there is none."""
    s, ts = oracle.scales(W, NVFP4, 16)
    x, w = oracle.normalise(W, NVFP4, 16, s, ts).astype(np.float64), np.broadcast_to(I.astype(np.float64), W.shape)
    T, most = T.astype(np.float64), None
    for r in range(rounds - 1):
        at = [np.searchsorted(0.5 * (t[1:] + t[:-1]), x) for t in T]
        err = [(w * (x - t[a]) ** 2).reshape(len(W), -1, 16).sum(-1) for t, a in zip(T, at)]
        cell = np.where(np.repeat(err[1] < err[0], 16, axis=1), at[1] + 16, at[0]).ravel()
        sw, sx = (np.bincount(cell, v.ravel(), minlength=32) for v in (w, w * x))
        if r == 2:
            most, about, q_most = sw, T.ravel().copy(), 0.0
        if r >= 2:
            q_most = max(q_most, (w.ravel() * (x.ravel() - about[cell]) ** 2).sum())
            if (sw <= 0.25 * most)[most > 0].any() or np.minimum(*err).sum() < 0.0625 * q_most:
                return r
            most = np.maximum(most, sw)
        T = np.sort(np.divide(sx, sw, out=T.ravel().copy(), where=sw > 0).reshape(2, 16), axis=1)
    return rounds - 1


@pytest.mark.parametrize("seed", [132, 163, 251, 21, 35, 46])
def test_sums_that_have_lost_their_accuracy_end_the_incremental_rounds(seed):
    """The first three: cells that grow behind the third round and shrink again, though never below a quarter of their
    weight there.  The others: an objective that falls far below its terms about the third round's tables."""
    rng = np.random.default_rng(seed)
    W = synth.f32_to_bf16_bits((rng.standard_normal((64, 512)) * 0.02).astype(np.float32))
    I = np.exp(rng.uniform(0.5, 3.0) * rng.standard_normal(512)).astype(np.float32)
    T01 = tables(*(np.linspace(*np.sort(rng.uniform(-6, 6, 2)), 16) for _ in range(2)))
    rounds = 28
    end = followed(W, I, T01, rounds)
    assert 3 < end < rounds - 1
    W = np.tile(W, (rows_for(24, 512) // 64, 1))
    ws = binding.alloc_workspace(NVFP4, *W.shape)
    o = oracle.fit_layer(W, NVFP4, 16, rounds, I=I, init="user", T_init=T01)
    r = binding.quantize_layer(dev_bf16(W), NVFP4, I=torch.from_numpy(I).cuda(), n_outer=rounds, init=binding.INIT_USER, ws=ws, want_trace=True,
                               T01_init=torch.from_numpy(T01))
    torch.cuda.synchronize()
    assert binding.debug_incremental(ws) == (3, end)
    assert int(r["status"].item()) == 0 and table_close(host(r["T01"]), o["T"])[0]
    assert np.allclose(host(r["trace"]), o["trace"], rtol=1e-5, atol=0)
    check_end_to_end_bits(r, o, f"seed {seed}")


@pytest.mark.parametrize("K,units,extra,rounds,inner", [(512, 20, 0, 29, 1), (1008, 20, 5, 29, 1), (4096, 28, -3, 25, 1), (512, 6, -3, 3, 14), (1008, 11, 5, 2, 10)])
def test_weight_sums_that_are_carried_are_exact(K, units, extra, rounds, inner):
    """The sums of I that the incremental passes start from, against 64-bit sums over the cells of the same tables: counts
    times importances, rounded a few dozen times to 2^-53.  (FP32 sums erred by 1e-8 in every cell.)"""
    N = rows_for(units, K) + extra
    W, X = layer(NVFP4, N, K, T=64, name=f"incremental/sums/{K}/{extra}", dist="student5")
    Wd, ws = dev_bf16(W), binding.alloc_workspace(NVFP4, N, K)
    r = binding.quantize_layer(Wd, NVFP4, X=dev_bf16(X), n_outer=rounds, n_inner=inner, init=binding.INIT_QUANTILE, ws=ws)
    torch.cuda.synchronize()
    assert binding.debug_incremental(ws)[0] == (3 if inner == 1 else 1)
    T, _, got = ws[272:272 + 768].clone().view(torch.float64).view(3, 2, 16)      # Ctrl::keep_T, keep_sx, keep_sw
    scale = torch.arange(128, dtype=torch.uint8, device="cuda").view(torch.float8_e4m3fn).float()[r["scales_pos"].long()] * r["tensor_scale"]
    I = r["I"].double().view(1, -1, 16)
    want = torch.zeros(2, 16, dtype=torch.float64, device="cuda")
    for r0 in range(0, N, 4096):
        x = (Wd[r0:r0 + 4096].float().view(-1, K // 16, 16) * (1.0 / scale[r0:r0 + 4096])[..., None]).double()
        cell = [torch.searchsorted((0.5 * (t[1:] + t[:-1])).contiguous(), x) for t in T]
        err = [(I * (x - t[c]) ** 2).sum(-1) for t, c in zip(T, cell)]
        second = (err[1] < err[0])[..., None]
        for t in range(2):
            mine = second if t else ~second
            for c in range(16):
                want[t, c] += (I * ((cell[t] == c) & mine)).sum()
    assert torch.allclose(got, want, rtol=1e-12, atol=0)


@pytest.mark.parametrize("rounds,inner,small", [(29, 1, False), (3, 10, False), (29, 1, True)])
def test_layers_that_share_a_launch(rounds, inner, small):
    """Two layers, each on its share of the blocks; with a small one in their launch all rounds of all three are full ones."""
    shapes = [(rows_for(12, 512), 512), (rows_for(14, 1008) + 5, 1008)] + [(70, 640)] * small
    cases, oracles = [], []
    for N, K in shapes:
        W, X = layer(NVFP4, N, K, T=64, name=f"incremental/batch/{K}")
        oracles.append(oracle.fit_layer(W, NVFP4, 16, rounds, X=X, n_inner=inner, init="quantile"))
        cases.append((W, oracles[-1]["I"]))
    for d, o in zip(run_fit_batch(cases, NVFP4, rounds, binding.INIT_QUANTILE, n_inner=inner), oracles):
        assert binding.debug_incremental(d["ws"]) == ((0, 0) if small else (3 if inner == 1 else 1, rounds * inner - 1))
        assert table_close(host(d["T01"]), o["T"])[0]
        assert np.allclose(host(d["err_trace"]), o["trace"], rtol=1e-5, atol=0)
        assert np.array_equal(host(d["scales"]), o["scales_unsigned"])


@pytest.mark.parametrize("K,units,extra,rounds,dist", [(512, 20, 0, 29, "normal"), (1008, 24, 5, 27, "student5"), (4096, 40, -3, 22, "student5")])
def test_objectives_behind_the_third_round_are_the_entries(K, units, extra, rounds, dist):
    """The objective of the incremental rounds and of the last, full one is that of the entries, not of the constants beside
    them (1e-7 of it): the FP32 roundings of millions of terms, 2^-24 each and of either sign, leave less than a sixth of one."""
    W, X = layer(NVFP4, rows_for(units, K) + extra, K, T=64, name=f"incremental/trace/{K}", dist=dist)
    o = oracle.fit_layer(W, NVFP4, 16, rounds, X=X, init="quantile")
    r = binding.quantize_layer(dev_bf16(W), NVFP4, X=dev_bf16(X), n_outer=rounds, init=binding.INIT_QUANTILE, want_trace=True)
    assert np.allclose(host(r["trace"])[3:], o["trace"][3:], rtol=1e-8, atol=0)


def test_two_runs_give_the_same_bits():
    N, K = rows_for(30, 2048), 2048
    W, X = layer(NVFP4, N, K, T=64, name="incremental/twice")
    out = []
    for _ in range(2):
        r = binding.quantize_layer(dev_bf16(W), NVFP4, X=dev_bf16(X), n_outer=25, init=binding.INIT_QUANTILE, want_trace=True)
        torch.cuda.synchronize()
        out.append([host(r[k]) for k in ("T01", "trace", "codes", "scales")])
    assert all(np.array_equal(a, b) for a, b in zip(*out))
