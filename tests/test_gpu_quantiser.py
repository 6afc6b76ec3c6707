"""GPU parity of the activation quantiser at its edges: remainders of the eight-value steps, tensors that are only 16-byte
aligned, quotients on rounding ties, maxima smaller than the data (clamping), scales outside the range of the reciprocal,
values that are not finite, and the launches that follow without a wait in between."""
import numpy as np
import pytest
import torch

import workloads as wl

pytestmark = pytest.mark.gpu


def _reference(Y, amax):
    """Eq. 5 with b = 8 in fp32: IEEE quotient, round half to even, clamp; a value that is not a number becomes 0."""
    s = np.float32(1.0) if amax == 0 else np.float32(amax) / np.float32(127.0)
    with np.errstate(all="ignore"):
        q = np.rint((Y / s).astype(np.float32))
    q = np.where(np.isnan(q), np.float32(0.0), q)
    return np.clip(q, -128, 127).astype(np.int8), s


def _run(Y, amax, offset):
    import paper_2206_15014_b200 as nm
    from gpu_util import DEV
    Yd = torch.empty(Y.size + offset, dtype=torch.float32, device=DEV)[offset:]
    Yd.copy_(torch.from_numpy(Y))
    a = torch.tensor([amax], dtype=torch.float32, device=DEV)
    sx = torch.zeros(1, dtype=torch.float32, device=DEV)
    Xq = torch.full((Y.size + 16,), 99, dtype=torch.int8, device=DEV)
    nm.nm_quantize_act(Yd, Y.size, a, Xq, sx)
    m = torch.zeros(1, dtype=torch.float32, device=DEV)
    nm.nm_absmax(Yd, Y.size, m)
    assert nm.nm_poll_status() == 0
    got = Xq.cpu().numpy()
    assert (got[Y.size:] == 99).all(), "written past the end"
    return got[:Y.size], sx.item(), m.item()


@pytest.mark.parametrize("count", [1, 7, 8, 9, 2047, 2048, 8191, 8193, 148 * 4 * 256 * 8 + 3, 148 * 4 * 256 * 32 + 21])
@pytest.mark.parametrize("offset", [0, 4])
def test_counts_and_alignment(count, offset):
    Y = wl.normal(np.random.default_rng(count), (count,))
    amax = np.abs(Y).max()
    got, sx, m = _run(Y, amax, offset)
    ref, s = _reference(Y, amax)
    assert m == amax and sx == s and np.array_equal(got, ref)


@pytest.mark.parametrize("amax", [127.0, 63.5, 1.0, 2.0 ** -140, 2.0 ** -118, 2.0 ** 126, 3.4e38, 0.0])
def test_ties_clamps_and_extreme_scales(amax):
    rng = np.random.default_rng(5)
    s = np.float32(amax) / np.float32(127.0) if amax else np.float32(1.0)
    half = (np.arange(-300, 300) * 0.5).astype(np.float32)
    with np.errstate(all="ignore"):
        near = np.concatenate([np.nextafter(half * s, np.float32(np.inf)), half * s, np.nextafter(half * s, np.float32(-np.inf))])
        Y = np.concatenate([near, half, half * 3e6, wl.normal(rng, (4000,)) * s * 60,
                            np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 3.4e38, -3.4e38, 1e-44], np.float32)]).astype(np.float32)
    got, sx, _ = _run(Y, np.float32(amax), 0)
    ref, s = _reference(Y, np.float32(amax))
    assert sx == s and np.array_equal(got, ref), np.nonzero(got != ref)[0][:10]


def test_back_to_back_with_the_linear_layer():
    """Maximum, quantiser and linear layer again and again on the same buffers, nothing waited for in between: every kernel may
    start while the one before it drains, and must still find its results."""
    import paper_2206_15014_b200 as nm
    from gpu_util import DEV, to_dev
    rng = np.random.default_rng(9)
    T, K = 200, 512
    W = wl.normal(rng, (K, K), 0.05)
    vb, mb = nm.nm_packed_sizes(K, K, 2, 4, 8)
    values = torch.zeros(vb, dtype=torch.uint8, device=DEV)
    meta = torch.zeros(mb // 4, dtype=torch.int32, device=DEV)
    scales = torch.zeros(K, dtype=torch.float32, device=DEV)
    nm.nm_project_pack(to_dev(W), None, K, K, 2, 4, 8, values, meta, scales)
    desc = nm.make_packed(K, K, 2, 4, 8, values, meta)
    h0 = to_dev(wl.normal(rng, (T, K)))

    def chain(wait):
        y, x = h0.clone(), torch.empty((T, K), dtype=torch.int8, device=DEV)
        amax, sx = torch.zeros(12, dtype=torch.float32, device=DEV), torch.zeros(12, dtype=torch.float32, device=DEV)
        for i in range(12):
            nm.nm_absmax(y, y.numel(), amax[i:])
            nm.nm_quantize_act(y, y.numel(), amax[i:], x, sx[i:])
            nm.nm_int_linear_dsx(x, T, desc, sx[i:], scales, None, y)
            if wait:
                torch.cuda.synchronize()
        return y, sx

    y_ref, sx_ref = chain(True)
    for _ in range(5):
        y, sx = chain(False)
        assert torch.equal(y, y_ref) and torch.equal(sx, sx_ref)
    nm.nm_debug_set_option("no_pdl", 1)  # every launch an ordinary one
    try:
        y, sx = chain(False)
    finally:
        nm.nm_debug_set_option("no_pdl", 0)
    assert torch.equal(y, y_ref) and torch.equal(sx, sx_ref)
