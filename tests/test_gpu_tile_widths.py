"""GPU parity of the one-CTA kernel at each of its token-tile widths (option "one_bn"), whatever its rule would pick: weights
in tensor-core form, sparse and dense, and weights rebuilt per stage, all four output kinds, against the CPU oracle bit for
bit.  Tokens end inside the second or a later tile, channels inside the second."""
import numpy as np
import pytest

import oracle
import workloads as wl

pytestmark = pytest.mark.gpu

CASES = [(bn, f) for f in ((2, 4, 8), (4, 4, 8)) for bn in (192, 128, 96, 64, 32)] + \
        [(bn, f) for f in ((2, 4, 4), (1, 4, 8), (2, 8, 4), (4, 8, 8), (4, 4, 4)) for bn in (192, 128, 64)]


@pytest.mark.parametrize("bn,fmt", CASES, ids=lambda v: str(v) if isinstance(v, int) else f"{v[0]}:{v[1]}-{v[2]}b")
@pytest.mark.parametrize("K,out", [(640, 208), (1152, 250)])  # rows that TMA can and cannot store
def test_width(bn, fmt, K, out):
    import paper_2206_15014_b200 as nm
    from gpu_util import PackedOnDevice, gpu_int_linear, gpu_int_linear_q8, gpu_int_linear_bf16
    n, m, bits = fmt
    oracle.set_threads(oracle.max_threads())
    rng = np.random.default_rng(bn + K)
    T = 2 * bn + 5
    W = wl.normal(rng, (out, K), 0.02)
    b = wl.normal(rng, (out,), 0.02)
    Xq, sx = oracle.quantize_act(wl.normal(rng, (T, K)))
    v, meta, s = oracle.project_pack(W, None, n, m, bits)
    acc_ref, Y_ref = oracle.int_linear(Xq, oracle.unpack(v, meta, out, K, n, m, bits), sx, s, b)
    packed = PackedOnDevice(v, meta, s, out, K, n, m, bits)
    sy = np.float32(np.abs(Y_ref).max()) / np.float32(100.0)
    for name, value in (("one_bn", bn), ("no_pair", 1), ("no_resident", 1)):
        nm.nm_debug_set_option(name, value)
    try:
        acc, Y = gpu_int_linear(Xq, packed, sx, b)
        q8, bf16 = gpu_int_linear_q8(Xq, packed, sx, b, sy), gpu_int_linear_bf16(Xq, packed, sx, b)
    finally:
        for name in ("one_bn", "no_pair", "no_resident"):
            nm.nm_debug_set_option(name, 0)
    assert np.array_equal(acc, acc_ref) and np.array_equal(Y, Y_ref)
    assert np.array_equal(q8, oracle.requantize_static(Y_ref, sy))
    assert np.array_equal(bf16, oracle.to_bf16(Y_ref))
