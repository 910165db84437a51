"""Inputs at the edges of what the entry points take: they are answered, or reported, and touch nothing else."""
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
