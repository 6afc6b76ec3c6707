"""GPU parity of the CTA-pair kernels for reductions of at most 1024 (2:4 and dense int8 weights) against the CPU oracle:
accumulators, fp32, int8 and bfloat16 outputs, bit for bit.  The option "xres" sends every shape to the kernel with resident
activations (1) or to the other pair kernel (2: resident 2:4 weights, streamed dense ones), however few tiles there are:
reductions that end inside a stage, one token, ragged token and output tiles, output rows that TMA cannot store, and runs of
tiles that cross token or output tiles inside a pair."""
import numpy as np
import pytest

import oracle
import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True, params=[1, 2], ids=["resident_activations", "other_pair_kernel"])
def kernel_choice(request):
    import paper_2206_15014_b200 as nm
    nm.nm_debug_set_option("xres", request.param)
    yield
    nm.nm_debug_set_option("xres", 0)


def _run(seed, T, K, out, n, bias=True):
    from gpu_util import PackedOnDevice, gpu_int_linear, gpu_int_linear_q8, gpu_int_linear_bf16
    oracle.set_threads(oracle.max_threads())
    rng = np.random.default_rng(seed)
    W = wl.normal(rng, (out, K), 0.02)
    b = wl.normal(rng, (out,), 0.02) if bias else None
    Xq, sx = oracle.quantize_act(wl.normal(rng, (T, K)))
    v, meta, s = oracle.project_pack(W, None, n, 4, 8)
    D = oracle.unpack(v, meta, out, K, n, 4, 8)
    acc_ref, Y_ref = oracle.int_linear(Xq, D, sx, s, b)
    packed = PackedOnDevice(v, meta, s, out, K, n, 4, 8)
    acc, Y = gpu_int_linear(Xq, packed, sx, b)
    assert np.array_equal(acc, acc_ref), f"{(acc != acc_ref).sum()} accumulators differ"
    assert np.array_equal(Y, Y_ref)
    sy = np.float32(np.abs(Y_ref).max()) / np.float32(100.0)
    assert np.array_equal(gpu_int_linear_q8(Xq, packed, sx, b, sy), oracle.requantize_static(Y_ref, sy))
    assert np.array_equal(gpu_int_linear_bf16(Xq, packed, sx, b), oracle.to_bf16(Y_ref))


# from 74 pair tiles on the library takes the pair kernels
@pytest.mark.parametrize("n", [2, 4])
@pytest.mark.parametrize("T,K,out", [
    (74 * 192, 128, 256),        # one tile per pair, the shortest reduction (half a 2:4 stage)
    (37 * 192 - 191, 640, 512),  # a last token tile of one token; a 2:4 reduction that ends inside a stage
    (3000, 1024, 1300),          # six output tiles, the last with 20 channels; runs that cross token tiles
    (5000, 768, 1002),           # rows of no output kind can be stored by TMA
    (4 * 192 + 5, 896, 4096),    # few token tiles, sixteen output tiles
    (14400, 256, 257),           # a second output tile of one channel
])
def test_shapes(T, K, out, n):
    _run(T + K, T, K, out, n)


@pytest.mark.parametrize("n", [2, 4])
def test_many_tiles_per_pair_no_bias(n):
    _run(5, 192 * 130 + 100, 384, 768, n, bias=False)


@pytest.mark.parametrize("n", [2, 4])
def test_library_choice_matches_the_other_pair_kernel(n):
    import torch
    import paper_2206_15014_b200 as nm
    from gpu_util import DEV
    T, K, out = 6000, 768, 2304
    g = torch.Generator(device=DEV).manual_seed(3)
    W = torch.randn((out, K), generator=g, device=DEV) * 0.02
    vb, mb = nm.nm_packed_sizes(out, K, n, 4, 8)
    values = torch.zeros(vb, dtype=torch.uint8, device=DEV)
    meta = torch.zeros(max(mb // 4, 1), dtype=torch.int32, device=DEV)
    scales = torch.zeros(out, dtype=torch.float32, device=DEV)
    nm.nm_project_pack(W, None, out, K, n, 4, 8, values, meta if n == 2 else None, scales)
    desc = nm.make_packed(out, K, n, 4, 8, values, meta if n == 2 else None)
    X = torch.randint(-128, 128, (T, K), generator=g, device=DEV, dtype=torch.int8)
    got = {}
    for choice in (0, 1, 2):
        nm.nm_debug_set_option("xres", choice)
        amax = torch.zeros(1, dtype=torch.float32, device=DEV)
        sx = torch.full((1,), 0.01, dtype=torch.float32, device=DEV)
        Y = torch.zeros((T, out), dtype=torch.float32, device=DEV)
        status = torch.zeros(1, dtype=torch.int32, device=DEV)
        nm.nm_int_linear_dsx(X, T, desc, sx, scales, None, Y, amax, status=status)
        assert nm.nm_poll_status(status) == nm.NM_OK
        assert amax.item() == Y.abs().max().item()
        got[choice] = Y
    assert torch.equal(got[0], got[1]) and torch.equal(got[0], got[2])
