"""The size-dependent branches of the library, at the sizes where they can go wrong, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_08692_b200 import binding, build, synth
from test_gpu_parity import DEV, INT4, NVFP4, check_end_to_end_bits, dev_bf16, host, layer, table_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


@pytest.mark.parametrize("mode,N,K", [
    (INT4, 512, 512),        # items of one row per warp
    (NVFP4, 1531, 2064),     # items of two rows, ragged rows and columns
    (INT4, 4003, 512),       # items of four rows, the last one ragged
    (NVFP4, 9479, 256),      # items of two rows, three per block (149 items of four would be one more than the blocks)
])
def test_rows_per_item(mode, N, K):
    W, X = layer(mode, N, K, name=f"items/{mode}/{N}x{K}")
    g = 128 if mode == INT4 else 16
    o = oracle.fit_layer(W, mode, g, 4, X=X, init="quantile")
    r = binding.quantize_layer(dev_bf16(W), mode, X=dev_bf16(X), n_outer=4, init=binding.INIT_QUANTILE, want_trace=True)
    torch.cuda.synchronize()
    assert int(r["status"].item()) == 0
    assert table_close(host(r["T01"]), o["T"])[0]
    assert np.allclose(host(r["trace"])[:4], o["trace"], rtol=1e-4, atol=0)
    check_end_to_end_bits(r, o, f"{mode} {N}x{K}")


@pytest.mark.parametrize("mode,extra", [(INT4, 1), (NVFP4, 1), (NVFP4, 0)])
def test_several_items_per_block(mode, extra):
    """Four items of four rows per block, the last one ragged; with one more than that, it is dealt out by quarters."""
    N, K = 64 * (4 * torch.cuda.get_device_properties(0).multi_processor_count + extra) - 5, 256
    test_rows_per_item(mode, N, K)


@pytest.mark.parametrize("mode", [INT4, NVFP4])
def test_rows_with_gaps(mode):
    """W as columns of a wider matrix: the start's passes find rows by division, the fit and pack passes by stride."""
    W, X = layer(mode, 67, 640, name=f"gaps/{mode}")
    wide = torch.zeros(67, 640 + 136, dtype=torch.bfloat16, device=DEV)
    wide[:, 64:704] = dev_bf16(W)
    g = 128 if mode == INT4 else 16
    o = oracle.fit_layer(W, mode, g, 3, X=X, init="quantile")
    r = binding.quantize_layer(wide[:, 64:704], mode, X=dev_bf16(X), n_outer=3, init=binding.INIT_QUANTILE)
    torch.cuda.synchronize()
    assert np.array_equal(host(r["scales_pos"]), o["scales_unsigned"])
    assert table_close(host(r["T01"]), o["T"])[0]
    check_end_to_end_bits(r, o, f"gaps {mode}")


@pytest.mark.parametrize("mode", [INT4, NVFP4])
def test_scales_over_the_whole_range_of_group_maxima(mode):
    """The scale rules replace a division by a product where rounding cannot tell them apart: every exponent from far
    below the smallest scale step to the layer's maximum, and mantissas next to half-way points, bit-exact."""
    g = 128 if mode == INT4 else 16
    rng = np.random.default_rng(5)
    groups = 1 << 16
    e = rng.integers(127 - 40, 128, groups) if mode == NVFP4 else rng.integers(20, 250, groups)
    top = (e << 7 | rng.integers(0, 128, groups)).astype(np.uint16)
    W = np.zeros((groups // 16, 16, g), np.uint16)
    W[:, :, 3] = top.reshape(-1, 16)
    W = W.reshape(groups // 16, 16 * g)
    want, ts = oracle.scales(W, mode, g)
    for init in (binding.INIT_GRID, binding.INIT_QUANTILE):        # the plain pass and the one that counts the histogram
        r = binding.quantize_layer(dev_bf16(W), mode, I=torch.ones(W.shape[1], device=DEV), n_outer=0, init=init,
                                   ws=binding.alloc_workspace(mode, *W.shape, full=True))
        torch.cuda.synchronize()
        assert np.array_equal(host(r["scales_pos"]), want) and host(r["tensor_scale"])[0] == ts[0]


@pytest.mark.parametrize("T", [64, 128, 129, 2049])
def test_importances_in_one_strip_and_in_several(T):
    K = 264
    X = synth.activations(T, K, 3, f"strips/{T}", kind="loguniform", massive_frac=0.01)
    I = torch.empty(K, dtype=torch.float32, device=DEV)
    binding.act_stats(dev_bf16(X), I, binding.alloc_workspace(NVFP4, 1, K))
    assert np.allclose(host(I), oracle.act_stats(X), rtol=1e-6, atol=0)      # one rounding to FP32: 2^-24


@pytest.mark.parametrize("mode,N,K,T", [(NVFP4, 1100, 2048, 65), (INT4, 255, 8192, 300), (NVFP4, 257, 8192, 1)])
def test_host_buffers_with_overlapped_copies(mode, N, K, T):
    """4 MB and more: copies on a stream of their own, rows packed in four ranges (the last one shorter)."""
    W, X = layer(mode, N, K, T=T, name=f"hostlanes/{mode}/{N}")
    g = 128 if mode == INT4 else 16
    pin = lambda *a, **k: torch.empty(*a, **k).pin_memory()
    out = dict(T01_host=pin(2, 16, dtype=torch.float32), T01_bf16_host=pin(2, 16, dtype=torch.int16),
               scales_host=pin(N, K // g, dtype=torch.int16 if mode == INT4 else torch.uint8), tensor_scale_host=pin(1, dtype=torch.float32),
               codes_host=pin(N, K // 2, dtype=torch.uint8), err_out_host=pin(2, dtype=torch.float64))
    ws = torch.empty(binding.host_workspace_bytes(mode, N, K, T), dtype=torch.uint8, device=DEV)
    binding.quantize_layer_host(torch.from_numpy(W.view(np.int16)).pin_memory(), torch.from_numpy(X.view(np.int16)).pin_memory(), mode,
                                n_outer=3, init=binding.INIT_QUANTILE, ws=ws, **out)
    o = oracle.fit_layer(W, mode, g, 3, X=X, init="quantile")
    assert table_close(out["T01_host"].numpy(), o["T"])[0]
    assert np.array_equal(out["T01_bf16_host"].numpy().view(np.uint16), o["T_bf16"])
    assert np.array_equal(out["codes_host"].numpy(), o["codes"])
    sc = out["scales_host"].numpy()
    assert np.array_equal(sc.view(np.uint16) if mode == INT4 else sc, o["scales"])
    assert np.isclose(out["err_out_host"][0].item(), o["E_final"], rtol=1e-4)


@pytest.mark.parametrize("mode,N,K", [(INT4, 9, 1024), (NVFP4, 31, 264 * 16), (NVFP4, 1, 16)])
def test_dequant_words_around_a_step(mode, N, K):
    """Four words of codes per thread and step: fewer, exactly as many and a few more, dense and with gaps between rows."""
    g = 128 if mode == INT4 else 16
    W, X = layer(mode, N, K, name=f"dq/{mode}/{N}")
    o = oracle.fit_layer(W, mode, g, 1, X=X, init="grid")
    want = oracle.dequant(o["codes"], o["scales"], o["tensor_scale"], o["T_bf16"], mode, g)
    u16 = lambda a: torch.from_numpy(a.view(np.int16)).to(DEV)
    args = (torch.from_numpy(o["codes"]).to(DEV), u16(o["scales"]) if mode == INT4 else torch.from_numpy(o["scales"]).to(DEV),
            torch.from_numpy(o["tensor_scale"]).to(DEV), u16(o["T_bf16"]), mode)
    for pad in (0, 24):
        buf = torch.full((N, K + pad), 7.0, dtype=torch.bfloat16, device=DEV)
        binding.dequant(*args, buf[:, :K])
        assert np.array_equal(host(buf[:, :K].contiguous()), want)
        assert bool((buf[:, K:] == 7.0).all())
