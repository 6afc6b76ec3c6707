"""GPU parity of the projection at the edges of its steps: rows that end inside a lane's eight columns or are only
16-byte aligned, groups of every shape that a cluster of blocks can and cannot hold, and batches whose launches overlap."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wl

pytestmark = pytest.mark.gpu


def _offset(a, floats):
    """`a` on the device at an address `floats` * 4 bytes past a 512-byte boundary."""
    from gpu_util import DEV
    t = torch.empty(a.size + floats, dtype=torch.float32, device=DEV)[floats:].view(a.shape)
    return t.copy_(torch.from_numpy(a))


def _buffers(out, k, n, m, bits):
    import paper_2206_15014_b200 as nm
    from gpu_util import DEV
    vb, mb = nm.nm_packed_sizes(out, k, n, m, bits)
    return (torch.full((vb + 16,), 0x5C, dtype=torch.uint8, device=DEV),
            torch.full((mb // 4 + 4,), 0x5C5C5C5C, dtype=torch.int32, device=DEV),
            torch.full((out,), -1.0, dtype=torch.float32, device=DEV), vb, mb)


def _same(bufs, ref):
    v, mt, sc, vb, mb = bufs
    vr, mr, sr = ref
    v, mt = v.cpu().numpy(), mt.cpu().numpy().view(np.uint32)
    assert np.array_equal(sc.cpu().numpy(), sr), "scales differ"
    assert np.array_equal(v[:vb], np.asarray(vr).reshape(-1)) and (v[vb:] == 0x5C).all()
    if mb:
        assert np.array_equal(mt[: mb // 4], np.asarray(mr).reshape(-1))
    assert (mt[mb // 4:] == 0x5C5C5C5C).all()


@pytest.mark.parametrize("n,m", [(2, 4), (1, 4), (4, 4), (1, 8), (2, 8), (4, 8)])
@pytest.mark.parametrize("bits", [8, 4])
def test_row_ends_and_alignment(n, m, bits):
    import paper_2206_15014_b200 as nm
    from gpu_util import DEV
    for i, (out, k) in enumerate([(7, 16), (9, 264), (5, 1028), (6, 2052), (3, 4092), (11, 776), (3, 4112)]):
        while k % m or (k // m * n * bits) % 8:  # whole groups and whole bytes of codes per row
            k += 4
        W, U = wl.pack_sweep_matrix(21, i, out, k)
        for off in (0, 4):  # 32-byte and 16-byte aligned operands
            Wd, Ud = _offset(W, off), _offset(U, off)
            for with_u in (False, True):
                bufs = _buffers(out, k, n, m, bits)
                status = torch.zeros(1, dtype=torch.int32, device=DEV)
                nm.nm_project_pack(Wd, Ud if with_u else None, out, k, n, m, bits, bufs[0], bufs[1] if n != m else None, bufs[2], status)
                assert nm.nm_poll_status(status) == nm.NM_OK
                _same(bufs, oracle.project_pack(W, U if with_u else None, n, m, bits))
            Z, Un = _offset(np.zeros_like(W), off), _offset(np.zeros_like(W), off)
            nm.nm_admm_project(Wd, Ud, out, k, n, m, bits, Z, Un, None, None, None, status)
            Zr, Unr, _ = oracle.admm_step(W, U, n, m, bits)
            assert np.array_equal(Z.cpu().numpy(), Zr) and np.array_equal(Un.cpu().numpy(), Unr)


@pytest.mark.parametrize("G", [1, 2, 3, 4, 5, 7, 11, 12, 16, 17, 24, 31, 32, 48, 64, 100, 128, 129])
@pytest.mark.parametrize("n,m,bits", [(2, 4, 4), (4, 8, 8), (1, 8, 4), (4, 4, 8)])
def test_group_sizes(n, m, bits, G):
    """One pass in a cluster where the group fits (4 to 128 warps, a suitable factor), two passes elsewhere; the last group short."""
    import paper_2206_15014_b200 as nm
    from gpu_util import DEV, to_dev
    for i, (out, k) in enumerate([(130, 768), (70, 1536), (45, 4096), (3, 1024), (33, 6144)]):
        W, U = wl.pack_sweep_matrix(22, i, out, k)
        W[out // 2] *= 20.0
        W[0] = 0.0
        ref = oracle.project_pack_grouped(W, U, n, m, bits, G)
        Wd, Ud = to_dev(W), to_dev(U)
        bufs = _buffers(out, k, n, m, bits)
        status = torch.zeros(1, dtype=torch.int32, device=DEV)
        nm.nm_project_pack_grouped(Wd, Ud, out, k, n, m, bits, G, bufs[0], bufs[1] if n != m else None, bufs[2], status)
        assert nm.nm_poll_status(status) == nm.NM_OK
        _same(bufs, ref)
        again = _buffers(out, k, n, m, bits)
        Z, Un = torch.empty_like(Wd), torch.empty_like(Wd)
        nm.nm_admm_project_grouped(Wd, Ud, out, k, n, m, bits, G, Z, Un, again[0], again[1] if n != m else None, again[2], status)
        assert nm.nm_poll_status(status) == nm.NM_OK
        _same(again, ref)
        D = oracle.unpack(ref[0], ref[1], out, k, n, m, bits)
        Zr = (ref[2][:, None] * D.astype(np.float32)).astype(np.float32)
        assert np.array_equal(Z.cpu().numpy(), Zr)
        assert np.array_equal(Un.cpu().numpy(), ((W + U).astype(np.float32) - Zr).astype(np.float32))


def test_overlapping_launches_of_a_batch_end_before_what_follows():
    """Six formats in one call: six launches of which each may start while the one before drains.  What comes next in the
    stream, a copy and a linear layer launched as a programmatic dependent, must find all of their outputs."""
    import paper_2206_15014_b200 as nm
    from gpu_util import DEV, to_dev
    fmts = [(2, 4, 8), (4, 4, 8), (1, 4, 8), (2, 4, 4), (4, 8, 8), (2, 8, 4)]
    shapes = [(4096, 1024), (96, 4096), (1000, 1024), (8, 1024), (700, 768), (64, 1024)]
    jobs, bufs, refs = [], [], []
    for i, ((n, m, bits), (out, k)) in enumerate(zip(fmts, shapes)):
        W, U = wl.pack_sweep_matrix(23, i, out, k)
        b = _buffers(out, k, n, m, bits)
        jobs.append((to_dev(W), to_dev(U), n, m, bits, b[0], b[1] if n != m else None, b[2]))
        bufs.append(b)
        refs.append(oracle.project_pack(W, U, n, m, bits))
    ws_bytes = nm.nm_pack_workspace_bytes(len(jobs))
    ws = torch.empty(ws_bytes, dtype=torch.uint8, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    X = torch.randint(-127, 128, (64, 1024), dtype=torch.int8, device=DEV)
    desc = nm.make_packed(4096, 1024, 2, 4, 8, bufs[0][0], bufs[0][1])
    ys = []
    for no_pdl in (0, 0, 1):
        nm.nm_debug_set_option("no_pdl", no_pdl)
        for b in bufs:
            b[0][: b[3]].fill_(0x11)
            b[2].fill_(-1.0)
        nm.nm_project_pack_batched(nm.make_pack_jobs(jobs), len(jobs), ws, ws_bytes, status)
        Y = torch.zeros((64, 4096), dtype=torch.float32, device=DEV)
        nm.nm_int_linear(X, 64, desc, 0.01, bufs[0][2], None, Y, status=status)
        copies = [(b[0].clone(), b[1].clone(), b[2].clone(), b[3], b[4]) for b in bufs]
        assert nm.nm_poll_status(status) == nm.NM_OK
        for c, r in zip(copies, refs):
            _same(c, r)
        ys.append(Y)
        nm.nm_debug_set_option("no_pdl", 0)
    assert torch.equal(ys[0], ys[1]) and torch.equal(ys[0], ys[2]) and ys[0].any()
    D = oracle.unpack(refs[0][0], refs[0][1], 4096, 1024, 2, 4, 8)
    _, Y_ref = oracle.int_linear(X.cpu().numpy(), D, np.float32(0.01), refs[0][2], None)
    assert np.array_equal(ys[0].cpu().numpy(), Y_ref)


def test_overlapping_group_launches_of_a_batch():
    """The same for group-wise scales: one cluster launch per format and row length, and a two-pass one (rows of 6144) among them."""
    import paper_2206_15014_b200 as nm
    from gpu_util import DEV, to_dev
    fmts = [(2, 4, 8), (4, 4, 8), (2, 4, 8), (2, 4, 4), (4, 8, 8), (2, 4, 8)]
    shapes = [(2000, 1024), (96, 4096), (100, 4096), (64, 6144), (700, 768), (33, 1536)]
    jobs, bufs, refs = [], [], []
    for i, ((n, m, bits), (out, k)) in enumerate(zip(fmts, shapes)):
        W, U = wl.pack_sweep_matrix(24, i, out, k)
        b = _buffers(out, k, n, m, bits)
        jobs.append((to_dev(W), to_dev(U), n, m, bits, b[0], b[1] if n != m else None, b[2]))
        bufs.append(b)
        refs.append(oracle.project_pack_grouped(W, U, n, m, bits, 32))
    ws_bytes = nm.nm_pack_workspace_bytes(len(jobs))
    ws = torch.empty(ws_bytes, dtype=torch.uint8, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    for _ in range(3):
        for b in bufs:
            b[0][: b[3]].fill_(0x11)
            b[2].fill_(-1.0)
        nm.nm_project_pack_grouped_batched(nm.make_pack_jobs(jobs), len(jobs), 32, ws, ws_bytes, status)
        copies = [(b[0].clone(), b[1].clone(), b[2].clone(), b[3], b[4]) for b in bufs]
        assert nm.nm_poll_status(status) == nm.NM_OK
        for c, r in zip(copies, refs):
            _same(c, r)


@pytest.mark.parametrize("kind", ["row", "group", "dist"])
def test_jobs_of_different_formats_on_one_dual_in_place_run_in_order(kind):
    """Three formats on the same W and U, the second one updating U in place: its launch must wait for the first, and the third
    reads what it wrote, as three calls of the one-matrix entry point do."""
    import paper_2206_15014_b200 as nm
    from gpu_util import DEV, to_dev
    out, k, G, ncand = 4096, 1024, 32, 4
    fmts = [(2, 4, 8), (4, 4, 4), (1, 4, 8)]
    single, batched, extra = {"row": (nm.nm_admm_project, nm.nm_admm_project_batched, ()),
                              "group": (nm.nm_admm_project_grouped, nm.nm_admm_project_grouped_batched, (G,)),
                              "dist": (nm.nm_admm_project_dist, nm.nm_admm_project_dist_batched, (ncand,))}[kind]
    W, U = wl.pack_sweep_matrix(25, 0, out, k)
    Wd, U0 = to_dev(W), to_dev(U * 8.0)
    ws_bytes = nm.nm_admm_workspace_bytes(len(fmts))
    ws = torch.empty(ws_bytes, dtype=torch.uint8, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)

    def buffers():
        Ud = U0.clone()
        return (Ud, [torch.zeros_like(Wd) for _ in fmts], [torch.zeros_like(Wd), Ud, torch.zeros_like(Wd)],
                [torch.zeros(out, dtype=torch.float32, device=DEV) for _ in fmts])

    Ud, Z_ref, Un_ref, s_ref = buffers()
    for i, f in enumerate(fmts):
        single(Wd, Ud, out, k, *f, *extra, Z_ref[i], Un_ref[i], None, None, s_ref[i], status)
        assert nm.nm_poll_status(status) == nm.NM_OK
    for _ in range(3):
        Ud, Z, Un, sc = buffers()
        jobs = nm.make_admm_jobs([(Wd, Ud, *f, Z[i], Un[i], None, None, sc[i]) for i, f in enumerate(fmts)])
        batched(jobs, len(fmts), *extra, ws, ws_bytes, status)
        assert nm.nm_poll_status(status) == nm.NM_OK
        for i in range(len(fmts)):
            assert torch.equal(sc[i], s_ref[i]) and torch.equal(Z[i], Z_ref[i]) and torch.equal(Un[i], Un_ref[i]), f"job {i}"
