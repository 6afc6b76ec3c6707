"""GPU parity of the kernel that splits a reduction over a cluster, in each of its forms (option "split"), against the CPU
oracle: accumulators, fp32, int8 and bfloat16 outputs, bit for bit.  k-blocks that do not divide evenly, rings that wrap,
the most k-blocks a CTA takes, one token, tokens that end inside a CTA's share, channels that end inside a tile."""
import numpy as np
import pytest

import oracle
import workloads as wl

pytestmark = pytest.mark.gpu

PLANS = [(2, 32), (4, 32), (2, 64), (4, 64), (8, 64), (2, 96), (4, 96), (2, 128), (4, 128), (8, 128)]


def _run(T, K, out, n, m=4, bits=8, plan=None):
    """plan: the split that must be taken; None: the library's choice, which must be one."""
    import paper_2206_15014_b200 as nm
    from gpu_util import PackedOnDevice, gpu_int_linear, gpu_int_linear_q8, gpu_int_linear_bf16
    taken = nm.nm_split_plan(T, out, K, n, m, bits)
    assert taken == plan if plan else taken > 1000
    oracle.set_threads(oracle.max_threads())
    rng = np.random.default_rng(T + K)
    W, b = wl.normal(rng, (out, K), 0.02), wl.normal(rng, (out,), 0.02)
    Xq, sx = oracle.quantize_act(wl.normal(rng, (T, K)))
    v, meta, s = oracle.project_pack(W, None, n, m, bits)
    acc_ref, Y_ref = oracle.int_linear(Xq, oracle.unpack(v, meta, out, K, n, m, bits), sx, s, b)
    packed = PackedOnDevice(v, meta, s, out, K, n, m, bits)
    acc, Y = gpu_int_linear(Xq, packed, sx, b)
    assert np.array_equal(acc, acc_ref), f"{(acc != acc_ref).sum()} accumulators differ"
    assert np.array_equal(Y, Y_ref)
    sy = np.float32(np.abs(Y_ref).max()) / np.float32(100.0)
    assert np.array_equal(gpu_int_linear_q8(Xq, packed, sx, b, sy), oracle.requantize_static(Y_ref, sy))
    assert np.array_equal(gpu_int_linear_bf16(Xq, packed, sx, b), oracle.to_bf16(Y_ref))


@pytest.mark.parametrize("n", [2, 4])
@pytest.mark.parametrize("splits,bn", PLANS)
def test_forms(splits, bn, n):
    import paper_2206_15014_b200 as nm
    nm.nm_debug_set_option("split", 1000 * splits + bn)
    try:
        _run(bn + bn // splits + 3, 128 * (splits + 1), 250, n, plan=1000 * splits + bn)  # one CTA has two k-blocks, the second token tile ends early
        if 9 * splits <= 64:
            _run(1, 128 * 9 * splits, 128, n, plan=1000 * splits + bn)                    # nine k-blocks in a ring of at most eight, one token
    finally:
        nm.nm_debug_set_option("split", 0)


@pytest.mark.parametrize("n,m,bits", [(2, 4, 4), (1, 4, 8), (1, 4, 4), (4, 8, 8), (4, 8, 4), (2, 8, 8), (1, 8, 4), (4, 4, 4)])
def test_formats_rebuilt_on_the_way(n, m, bits):
    import paper_2206_15014_b200 as nm
    try:
        for splits, bn in ((2, 32), (4, 64), (8, 128)):
            nm.nm_debug_set_option("split", 1000 * splits + bn)
            _run(bn + bn // splits + 3, 128 * (splits + 1), 250, n, m, bits, 1000 * splits + bn)
            if splits < 8:
                _run(1, 128 * 9 * splits, 128, n, m, bits, 1000 * splits + bn)
        nm.nm_debug_set_option("split", 0)
        for T, K, out in ((5, 1024, 1024), (130, 768, 770), (64, 4096, 300)):  # the library's choice: split
            _run(T, K, out, n, m, bits)
    finally:
        nm.nm_debug_set_option("split", 0)


@pytest.mark.parametrize("n", [2, 4])
@pytest.mark.parametrize("T,K,out", [(64, 8192, 384), (384, 4096, 1024), (128, 768, 768), (7, 512, 100), (700, 3072, 770)])
def test_library_choice_matches_the_unsplit_kernel(T, K, out, n):
    import torch
    import paper_2206_15014_b200 as nm
    from gpu_util import DEV
    g = torch.Generator(device=DEV).manual_seed(K)
    W = torch.randn((out, K), generator=g, device=DEV) * 0.02
    vb, mb = nm.nm_packed_sizes(out, K, n, 4, 8)
    values, scales = torch.zeros(vb, dtype=torch.uint8, device=DEV), torch.zeros(out, device=DEV)
    meta = torch.zeros(max(mb // 4, 1), dtype=torch.int32, device=DEV) if n == 2 else None
    nm.nm_project_pack(W, None, out, K, n, 4, 8, values, meta, scales)
    desc = nm.make_packed(out, K, n, 4, 8, values, meta)
    X = torch.randint(-128, 128, (T, K), generator=g, device=DEV, dtype=torch.int8)
    got = []
    for choice in (0, 1, 2128):
        nm.nm_debug_set_option("split", choice)
        taken = nm.nm_split_plan(T, out, K, n, 4, 8)
        assert taken == (0 if choice == 1 else choice) if choice else taken > 1000
        amax, sx = torch.zeros(1, device=DEV), torch.full((1,), 0.01, device=DEV)
        Y, status = torch.zeros((T, out), device=DEV), torch.zeros(1, dtype=torch.int32, device=DEV)
        try:
            nm.nm_int_linear_dsx(X, T, desc, sx, scales, None, Y, amax, status=status)
        finally:
            nm.nm_debug_set_option("split", 0)
        assert nm.nm_poll_status(status) == nm.NM_OK
        assert amax.item() == Y.abs().max().item()
        got.append(Y)
    assert torch.equal(got[0], got[1]) and torch.equal(got[0], got[2])


def test_a_split_that_does_not_fit_is_refused():
    import torch
    import paper_2206_15014_b200 as nm
    t = torch.zeros(1 << 22, dtype=torch.uint8, device="cuda")
    desc = nm.make_packed(770, 3072, 2, 4, 8, t, t)
    try:
        for forced in (2064, 8192, 7):  # 154 CTAs; no such width; no such number of CTAs
            nm.nm_debug_set_option("split", forced)
            with pytest.raises(nm.NmError) as e:
                nm.nm_int_linear(t, 700, desc, 1.0, t, None, t)
            assert e.value.code == nm.NM_ERR_UNSUPPORTED
    finally:
        nm.nm_debug_set_option("split", 0)
