"""GPU parity: int8 (static scale, Eq. 5 with b = 8) and bfloat16 outputs of the N:M integer linear layer.

Both sides form y with the same three fp32 operations (int -> float, one multiply for sx * sw[o], one
fma with the bias), divide by the scale with an IEEE division and round half to even, so the int8 codes
and the bfloat16 bit patterns are compared bit for bit.
"""
import numpy as np
import pytest

import oracle
import workloads as wl

pytestmark = pytest.mark.gpu

# int8 2:4 and dense (TMA weights, CTA pairs when large), and weights rebuilt in shared memory
MODES = [(2, 4, 8), (4, 4, 8), (2, 4, 4), (1, 4, 8), (2, 8, 8), (4, 8, 8)]
# (tokens, K, out): one tile; ragged, out % 16 != 0 (plain stores) ; out % 16 == 0 but ragged tokens;
# many tiles of a short reduction (CTA pairs) with output-tile changes; long reduction with streamed weights
# the last one: CTA pairs with rows that no TMA store can address (plain stores from sixteen warps)
# (the pair kernels for short reductions one by one: test_gpu_xres.py)
SHAPES = [(64, 128, 128), (100, 384, 200), (77, 256, 208), (4096 + 37, 512, 1280), (6000 + 3, 2048, 640), (7680 + 5, 512, 516)]


def _setup(seed, T, K, out, n, m, bits):
    rng = np.random.default_rng(seed)
    W = wl.normal(rng, (out, K), 0.02)
    b = wl.normal(rng, (out,), 0.02)
    X = wl.normal(rng, (T, K))
    Xq, sx = oracle.quantize_act(X)
    v, meta, s = oracle.project_pack(W, None, n, m, bits)
    D = oracle.unpack(v, meta, out, K, n, m, bits)
    oracle.set_threads(oracle.max_threads())
    _, Y = oracle.int_linear(Xq, D, sx, s, b, want_acc=False)
    return Xq, sx, v, meta, s, b, Y


@pytest.mark.parametrize("n,m,bits", MODES)
@pytest.mark.parametrize("T,K,out", SHAPES)
def test_int8_output_matches_oracle(n, m, bits, T, K, out):
    from gpu_util import PackedOnDevice, gpu_int_linear_q8
    Xq, sx, v, meta, s, b, Y = _setup(21, T, K, out, n, m, bits)
    packed = PackedOnDevice(v, meta, s, out, K, n, m, bits)
    amax = np.float32(np.abs(Y).max())
    for sy in (amax / np.float32(127.0), amax / np.float32(40.0)):  # full range; two thirds of the outputs clamp
        ref = oracle.requantize_static(Y, sy)
        got = gpu_int_linear_q8(Xq, packed, sx, b, sy)
        assert np.array_equal(got, ref), f"{(got != ref).sum()} of {ref.size} codes differ at sy={sy}"


@pytest.mark.parametrize("n,m,bits", MODES)
@pytest.mark.parametrize("T,K,out", SHAPES)
def test_bf16_output_matches_oracle(n, m, bits, T, K, out):
    from gpu_util import PackedOnDevice, gpu_int_linear_bf16
    Xq, sx, v, meta, s, b, Y = _setup(22, T, K, out, n, m, bits)
    got = gpu_int_linear_bf16(Xq, PackedOnDevice(v, meta, s, out, K, n, m, bits), sx, b)
    ref = oracle.to_bf16(Y)
    assert np.array_equal(got, ref), f"{(got != ref).sum()} of {ref.size} patterns differ"


def test_int8_chain_of_two_layers():
    # layer 1 writes int8 with a static scale; layer 2 consumes it as its X with sx = that scale
    from gpu_util import PackedOnDevice, gpu_int_linear, gpu_int_linear_q8
    T, K, H, out = 1000, 768, 3072, 768
    rng = np.random.default_rng(23)
    W1, b1 = wl.normal(rng, (H, K), 0.02), wl.normal(rng, (H,), 0.02)
    W2, b2 = wl.normal(rng, (out, H), 0.02), wl.normal(rng, (out,), 0.02)
    Xq, sx = oracle.quantize_act(wl.normal(rng, (T, K)))
    v1, m1, s1 = oracle.project_pack(W1, None, 2, 4, 8)
    v2, m2, s2 = oracle.project_pack(W2, None, 2, 4, 4)
    oracle.set_threads(oracle.max_threads())
    _, Y1 = oracle.int_linear(Xq, oracle.unpack(v1, m1, H, K, 2, 4, 8), sx, s1, b1, want_acc=False)
    sy = np.float32(np.abs(Y1).max()) / np.float32(127.0)
    H1 = oracle.requantize_static(Y1, sy)
    acc2, Y2 = oracle.int_linear(H1, oracle.unpack(v2, m2, out, H, 2, 4, 4), sy, s2, b2)
    g1 = gpu_int_linear_q8(Xq, PackedOnDevice(v1, m1, s1, H, K, 2, 4, 8), sx, b1, sy)
    assert np.array_equal(g1, H1)
    gacc2, gY2 = gpu_int_linear(g1, PackedOnDevice(v2, m2, s2, out, H, 2, 4, 4), sy, b2)
    assert np.array_equal(gacc2, acc2) and np.array_equal(gY2, Y2)


@pytest.mark.parametrize("T,K,out", [(300, 4096, 128), (8960, 1024, 512), (8960, 4096, 512)])
@pytest.mark.parametrize("n,m,bits", [(2, 4, 8), (4, 4, 8), (2, 4, 4)])
def test_accumulators_from_zero_to_the_largest(n, m, bits, T, K, out):
    """Constant rows of X against all-ones weights give every token its own accumulator value, from 0 up to the
    largest the operands allow (beyond 2^22 and 2^24 in magnitude for 8-bit codes, where int -> float rounds): fp32,
    int8 and bfloat16 outputs bit for bit on the one-CTA kernel, the pair kernels for short reductions and the 512-channel one."""
    from gpu_util import PackedOnDevice, gpu_int_linear, gpu_int_linear_q8, gpu_int_linear_bf16
    oracle.set_threads(oracle.max_threads())
    W = np.ones((out, K), np.float32)
    b = wl.normal(np.random.default_rng(31), (out,), 0.5)
    v, meta, s = oracle.project_pack(W, None, n, m, bits)
    D = oracle.unpack(v, meta, out, K, n, m, bits)
    c = ((np.arange(T) * 37) % 256 - 128).astype(np.int8)
    Xq = np.repeat(c[:, None], K, axis=1)
    sx = np.float32(2e-4)
    acc_ref, Y = oracle.int_linear(Xq, D, sx, s, b)
    if bits == 8:
        assert np.abs(acc_ref).max() > (1 << 22)
    packed = PackedOnDevice(v, meta, s, out, K, n, m, bits)
    acc, Yg = gpu_int_linear(Xq, packed, sx, b)
    assert np.array_equal(acc, acc_ref) and np.array_equal(Yg, Y)
    sy = np.float32(np.abs(Y).max()) / np.float32(127.0)
    assert np.array_equal(gpu_int_linear_q8(Xq, packed, sx, b, sy), oracle.requantize_static(Y, sy))
    assert np.array_equal(gpu_int_linear_bf16(Xq, packed, sx, b), oracle.to_bf16(Y))


def test_narrow_outputs_reject_bad_arguments():
    import torch
    import paper_2206_15014_b200 as nm
    from gpu_util import PackedOnDevice, to_dev
    rng = np.random.default_rng(24)
    v, meta, s = oracle.project_pack(wl.normal(rng, (128, 128), 0.02), None, 2, 4, 8)
    packed = PackedOnDevice(v, meta, s, 128, 128, 2, 4, 8)
    X = to_dev(np.zeros((16, 128), np.int8))
    Yq = torch.zeros((16, 128), dtype=torch.int8, device="cuda")
    for bad in (0.0, -1.0, float("inf"), float("nan")):
        with pytest.raises(nm.NmError):
            nm.nm_int_linear_q8(X, 16, packed.desc, 1.0, packed.scales, None, bad, Yq)
    with pytest.raises(nm.NmError):
        nm.nm_int_linear_q8(X, 16, packed.desc, 1.0, packed.scales, None, 1.0, None)
    with pytest.raises(nm.NmError):
        nm.nm_int_linear_bf16(X, 16, packed.desc, 1.0, None, None, Yq)
    with pytest.raises(nm.NmError):  # bfloat16 output on an odd byte address
        buf = torch.zeros(16 * 128 * 2 + 2, dtype=torch.uint8, device="cuda")
        nm.nm_int_linear_bf16(X, 16, packed.desc, 1.0, packed.scales, None, buf[1:], None)


# (tokens, K, out, n, m, bits, options): every kernel that stores int8 tiles, and the split one
SCALE_CASES = [
    (77, 128, 208, 2, 4, 8, {"split": 1}),         # one-CTA kernel, weights through TMA
    (77, 256, 208, 4, 4, 8, {"split": 2032}),      # split reduction: stores of its own
    (4096 + 37, 512, 1280, 2, 4, 4, {}),           # one-CTA kernel, weights rebuilt and resident
    (300, 2048, 640, 1, 8, 4, {"split": 1}),       # ... rebuilt for every k-block
    (3000, 1024, 1296, 2, 4, 8, {"xres": 1}),      # pair kernel with resident activations
    (3000, 1024, 1296, 4, 4, 8, {"xres": 1}),
    (3000, 1024, 1296, 2, 4, 8, {"xres": 2}),      # ... with resident weights
    (6003, 2048, 640, 4, 4, 8, {}),                # ... with both streamed
    (6003, 2048, 640, 2, 4, 8, {"no_wide": 1}),
    (6003, 2048, 640, 2, 4, 8, {}),                # 512-channel kernel
    (6003, 2048, 640, 2, 4, 4, {}),
]


@pytest.mark.parametrize("T,K,out,n,m,bits,options", SCALE_CASES)
def test_int8_output_at_any_scale(T, K, out, n, m, bits, options):
    """Quotients y / sy from far inside one code to far beyond the integers that single precision holds, both signs: every
    power of two around 2^23, where codes taken from bits of a sum could leave their range, and 1e-9 to 1e9 of the largest |Y|."""
    import paper_2206_15014_b200 as nm
    from gpu_util import PackedOnDevice, gpu_int_linear_q8
    Xq, sx, v, meta, s, b, Y = _setup(T + K, T, K, out, n, m, bits)
    packed = PackedOnDevice(v, meta, s, out, K, n, m, bits)
    amax = np.float32(np.abs(Y).max())
    try:
        for k, x in options.items():
            nm.nm_debug_set_option(k, x)
        for quotient in [2.0 ** e for e in range(20, 29)] + [1e9, 1e-9, 1e5, 1e36]:
            sy = np.float32(float(amax) / quotient)
            ref = oracle.requantize_static(Y, sy)
            got = gpu_int_linear_q8(Xq, packed, sx, b, sy)
            assert np.array_equal(got, ref), f"{(got != ref).sum()} of {ref.size} codes differ at max|Y| / sy = {quotient}"
    finally:
        for k in options:
            nm.nm_debug_set_option(k, 0)


# every kernel that has both forms of bfloat16 tiles: the last token unit is cut short, the last 128 channels too
@pytest.mark.parametrize("K,n,m,bits,options", [
    (1152, 4, 4, 8, {}),            # pair kernel with eight epilogue warps, weights streamed
    (1024, 2, 4, 8, {"xres": 2}),   # ... with sixteen, weights resident
    (768, 2, 4, 8, {"xres": 1}),    # resident activations
    (896, 4, 4, 8, {"xres": 1}),
    (1024, 2, 4, 4, {}),            # one-CTA kernel, weights rebuilt and resident, sparse and dense form
    (768, 4, 8, 4, {}),
])
@pytest.mark.parametrize("grouped", [1, 2])
def test_bfloat16_tiles_shared_or_own(K, n, m, bits, options, grouped):
    import paper_2206_15014_b200 as nm
    from gpu_util import PackedOnDevice, gpu_int_linear_bf16
    T, out = 2900, 1288
    Xq, sx, v, meta, s, b, Y = _setup(K, T, K, out, n, m, bits)
    packed = PackedOnDevice(v, meta, s, out, K, n, m, bits)
    options = dict(options, grouped=grouped)
    try:
        for k, x in options.items():
            nm.nm_debug_set_option(k, x)
        assert np.array_equal(gpu_int_linear_bf16(Xq, packed, sx, b), oracle.to_bf16(Y))
    finally:
        for k in options:
            nm.nm_debug_set_option(k, 0)


@pytest.mark.parametrize("n,m,bits,out", [(2, 4, 8, 3072), (2, 4, 4, 3080), (4, 4, 8, 3080), (2, 8, 4, 3072)])
def test_bfloat16_too_large_for_the_cache(n, m, bits, out):
    """At 192 MB of Y the pair kernels, and the one-CTA kernel with resident weights, store whole lines, shared by four warps: the same
    bits as pieces of the same tokens, which do not."""
    import torch
    import paper_2206_15014_b200 as nm
    from gpu_util import DEV
    T, K = 34000, 1024  # the last tile ends inside a unit of 16 tokens
    g = torch.Generator(device=DEV).manual_seed(out)
    W = torch.randn((out, K), generator=g, device=DEV) * 0.02
    vb, mb = nm.nm_packed_sizes(out, K, n, m, bits)
    values, scales = torch.zeros(vb, dtype=torch.uint8, device=DEV), torch.zeros(out, device=DEV)
    meta = torch.zeros(mb // 4, dtype=torch.int32, device=DEV) if n != m else None
    nm.nm_project_pack(W, None, out, K, n, m, bits, values, meta, scales)
    desc = nm.make_packed(out, K, n, m, bits, values, meta)
    X = torch.randint(-128, 128, (T, K), generator=g, device=DEV, dtype=torch.int8)
    Y, P = (torch.zeros((T, out), dtype=torch.bfloat16, device=DEV) for _ in range(2))
    nm.nm_int_linear_bf16(X, T, desc, 0.02, scales, None, Y)
    for a in range(0, T, 5000):
        b = min(T, a + 5000)
        nm.nm_int_linear_bf16(X[a:b], b - a, desc, 0.02, scales, None, P[a:b])
    assert torch.equal(Y.view(torch.int16), P.view(torch.int16))
    assert Y.any()
