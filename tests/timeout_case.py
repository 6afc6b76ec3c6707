"""Child process of test_gpu_timeout.py: runs against the library built with short device-side wait limits and the
skipped-stage test hook (NMSPARSE_LIB points at it).  For one kernel family per invocation: a launch whose CTA 0 never
issues one pipeline stage must come back with NM_ERR_TIMEOUT (no hang, no fault, context usable), and a normal launch
on the same stream right afterwards must match the CPU oracle.  Prints "ok <family>" on success."""
import os
import sys

import numpy as np
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import oracle  # noqa: E402
import workloads as wl  # noqa: E402
import paper_2206_15014_b200 as nm  # noqa: E402

# family -> (tokens, K, out, weight bits, options, int8 output?)
FAMILIES = {
    "one_cta": (64, 512, 128, 8, {"split": 1}, False),             # one tile, four stages, nm_gemm_kernel
    "one_cta_narrow": (64, 512, 128, 8, {"split": 1}, True),       # the same with int8 outputs (staging tiles of each warp's own)
    "pair": (74 * 192, 1024, 256, 8, {}, False),                   # one tile of four stages per SM pair, resident weights: pair 0 stalls alone
    "pair_streamed": (74 * 192, 1024, 256, 8, {"no_resident": 1}, False),
    "split": (64, 4096, 128, 8, {"split": 4064}, False),           # one tile over a cluster of four CTAs, eight stages each: CTA 0 stalls alone
    "split_rebuilt": (32, 6144, 128, 4, {"split": 2032}, False),   # ... of two, 24 stages in a shorter ring, weights built on the way
}


def pack_staged():
    """The staged projection kernel: warp 0 of block 0 never issues the copies of its second unit; its wait for that
    chunk expires, the launch reports the time-out, the next call is right."""
    dev = torch.device("cuda:0")
    oracle.set_threads(oracle.max_threads())
    out, k = 2048, 1024                       # 512 units: block 0 of the 444 resident blocks takes units 0 and 444
    W, U = wl.pack_sweep_matrix(5, 0, out, k)
    v_ref, meta_ref, s_ref = oracle.project_pack(W, U, 2, 4, 8)
    td = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)
    Wd, Ud = td(W), td(U)
    vb, mb = nm.nm_packed_sizes(out, k, 2, 4, 8)
    status = torch.zeros(1, dtype=torch.int32, device=dev)

    def launch():
        values = torch.zeros(vb, dtype=torch.uint8, device=dev)
        meta = torch.zeros(mb // 4, dtype=torch.int32, device=dev)
        scales = torch.zeros(out, dtype=torch.float32, device=dev)
        nm.nm_project_pack(Wd, Ud, out, k, 2, 4, 8, values, meta, scales, status)
        return values, meta, scales

    nm.nm_debug_set_option("pack_form", 2)
    nm.nm_debug_set_option("skip_pack_copy", 2)
    launch()
    rc = nm.nm_poll_status(status)
    assert rc == nm.NM_ERR_TIMEOUT, f"expected a timeout, got {nm.nm_strerror(rc)} {nm.nm_last_cuda_error()}"
    nm.nm_debug_set_option("skip_pack_copy", 0)
    status.zero_()
    values, meta, scales = launch()
    rc = nm.nm_poll_status(status)
    assert rc == nm.NM_OK, nm.nm_strerror(rc)
    assert np.array_equal(values.cpu().numpy().reshape(v_ref.shape), v_ref)
    assert np.array_equal(meta.cpu().numpy().view(np.uint32).reshape(meta_ref.shape), meta_ref)
    assert np.array_equal(scales.cpu().numpy(), s_ref), "the call after the timeout does not match the oracle"
    print("ok pack_staged")


def main(family):
    if family == "pack_staged":
        return pack_staged()
    T, K, out, bits, options, narrow = FAMILIES[family]
    dev = torch.device("cuda:0")
    oracle.set_threads(oracle.max_threads())
    rng = np.random.default_rng(7)
    W = wl.normal(rng, (out, K), 0.02)
    b = wl.normal(rng, (out,), 0.02)
    Xq, sx = oracle.quantize_act(wl.normal(rng, (T, K)))
    v, meta, s = oracle.project_pack(W, None, 2, 4, bits)
    D = oracle.unpack(v, meta, out, K, 2, 4, bits)
    _, Y_ref = oracle.int_linear(Xq, D, sx, s, b, want_acc=False)
    sy = np.float32(np.abs(Y_ref).max()) / np.float32(127.0)
    td = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)
    Xd, vd, md, sd, bd = td(Xq), td(v.reshape(-1)), td(meta.reshape(-1).view(np.int32)), td(s), td(b)
    desc = nm.make_packed(out, K, 2, 4, bits, vd, md)
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    for k_, v_ in options.items():
        nm.nm_debug_set_option(k_, v_)

    def launch():
        if narrow:
            Y = torch.zeros((T, out), dtype=torch.int8, device=dev)
            nm.nm_int_linear_q8(Xd, T, desc, float(sx), sd, bd, float(sy), Y, status=status)
        else:
            Y = torch.zeros((T, out), dtype=torch.float32, device=dev)
            nm.nm_int_linear(Xd, T, desc, float(sx), sd, bd, Y, status=status)
        return Y

    nm.nm_debug_set_option("skip_stage", 2)   # CTA 0 never issues its second pipeline stage
    Y = launch()
    rc = nm.nm_poll_status(status)
    assert rc == nm.NM_ERR_TIMEOUT, f"expected a timeout, got {nm.nm_strerror(rc)} {nm.nm_last_cuda_error()}"
    if family.startswith("split"):            # the cluster's other CTAs know: nobody writes sums that lack a part
        assert not Y.any()
    nm.nm_debug_set_option("skip_stage", 0)
    status.zero_()
    Y = launch()                              # same stream, same context: a normal call works and is right
    rc = nm.nm_poll_status(status)
    assert rc == nm.NM_OK, nm.nm_strerror(rc)
    ref = oracle.requantize_static(Y_ref, sy) if narrow else Y_ref
    assert np.array_equal(Y.cpu().numpy(), ref), "the call after the timeout does not match the oracle"
    print("ok", family)


if __name__ == "__main__":
    main(sys.argv[1])
