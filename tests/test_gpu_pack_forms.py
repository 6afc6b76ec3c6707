"""GPU parity of the projection kernel's two forms in blocks of four warps, each forced in turn, and at the sizes where
the library changes from one to the other.

"direct" (one unit per block, loads straight into registers) exists for every pattern, code width and output, with two register
budgets.  "staged" (persistent, the next rows brought into shared memory by bulk copies) exists for 1:4, 2:4, 1:8 and 2:8 without
dense outputs; the library takes it for launches with two operands and rows of 1024, 2048 or 4096 weights (2:4: of a multiple of
1024) of more than one round of the direct form's resident blocks, several matrices up to six.
Rows of one and four warps, ragged tails, a launch of many rounds per resident block, a batch through the device job
table, and (direct) the ADMM step with dense outputs, bit for bit against the oracle.
"""
import numpy as np
import pytest
import torch

import oracle
import workloads as wl

pytestmark = pytest.mark.gpu

PATTERNS = [(1, 4), (2, 4), (1, 8), (2, 8), (4, 8), (4, 4)]
STAGED = [(1, 4), (2, 4), (1, 8), (2, 8)]
FORMS = {"direct": 1, "staged": 2}


@pytest.fixture
def form(request):
    import paper_2206_15014_b200 as nm
    nm.nm_debug_set_option("pack_form", FORMS[request.param])
    yield request.param
    nm.nm_debug_set_option("pack_form", 0)


def _check_pack(W, U, n, m, bits):
    from gpu_util import gpu_project_pack
    v, meta, s, rc = gpu_project_pack(W, U, n, m, bits)
    v_ref, meta_ref, s_ref = oracle.project_pack(W, U, n, m, bits)
    assert rc == 0
    assert np.array_equal(s, s_ref), "scales differ"
    assert np.array_equal(v, v_ref), f"values differ in {(v != v_ref).sum()} bytes"
    if n != m:
        assert np.array_equal(meta, meta_ref), "metadata differs"


@pytest.mark.parametrize("form,n,m", [("direct", *p) for p in PATTERNS] + [("staged", *p) for p in STAGED], indirect=["form"])
@pytest.mark.parametrize("bits", [8, 4])
def test_forms_rows_and_ragged(form, n, m, bits):
    oracle.set_threads(oracle.max_threads())
    for seed, (out, k) in enumerate([(260, 1024), (70, 4096), (37, 3072)]):
        W, U = wl.pack_sweep_matrix(3, seed, out, k)
        _check_pack(W, U, n, m, bits)
    for seed, (out, k) in enumerate([(5, 8), (9, 1032), (6, 2072)]):
        if (k // m * n * bits) % 8:
            k *= 2
        _check_pack(wl.tie_heavy(100 + seed, out, k), None, n, m, bits)
        _check_pack(wl.with_outliers(110 + seed, out, k), wl.tie_heavy(120 + seed, out, k, levels=1), n, m, bits)


@pytest.mark.parametrize("form,n,m,bits", [("staged", 2, 4, 8), ("staged", 1, 4, 4), ("staged", 2, 8, 8), ("staged", 1, 8, 4), ("direct", 2, 4, 8), ("direct", 4, 8, 4), ("direct", 1, 8, 8)],
                         indirect=["form"])
def test_forms_many_rounds(form, n, m, bits):
    """More units than resident blocks, several times over (9001 rows of 1024: 2251 units; 1500 rows of 3072: a row
    spans four warps, one of them past the row's end), with the last block's rows running out."""
    oracle.set_threads(oracle.max_threads())
    for seed, (out, k) in enumerate([(9001, 1024), (1500, 3072)]):
        W, U = wl.pack_sweep_matrix(11, seed, out, k)
        _check_pack(W, U, n, m, bits)


@pytest.mark.parametrize("form", sorted(FORMS), indirect=True)
def test_forms_batched_through_the_job_table(form):
    """Twelve matrices of mixed shapes in one launch (device job table): a block's consecutive units cross from one
    job into the next."""
    import paper_2206_15014_b200 as nm
    from gpu_util import DEV, to_dev
    shapes = [(96, 1024), (40, 4096), (64, 1024), (700, 1024), (50, 768), (330, 2048)] * 2
    n, m, bits = 2, 4, 8
    jobs, refs = [], []
    for i, (out, k) in enumerate(shapes):
        W, U = wl.pack_sweep_matrix(17, i, out, k)
        vb, mb = nm.nm_packed_sizes(out, k, n, m, bits)
        bufs = (torch.zeros(vb, dtype=torch.uint8, device=DEV), torch.zeros(mb // 4, dtype=torch.int32, device=DEV),
                torch.zeros(out, dtype=torch.float32, device=DEV))
        jobs.append((to_dev(W), to_dev(U) if i % 2 == 0 else None, n, m, bits, *bufs))
        refs.append(oracle.project_pack(W, U if i % 2 == 0 else None, n, m, bits))
    arr = nm.make_pack_jobs(jobs)
    ws_bytes = nm.nm_pack_workspace_bytes(len(jobs))
    ws = torch.empty(ws_bytes, dtype=torch.uint8, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    nm.nm_project_pack_batched(arr, len(jobs), ws, ws_bytes, status)
    assert nm.nm_poll_status(status) == 0
    for job, (v_ref, m_ref, s_ref) in zip(jobs, refs):
        assert np.array_equal(job[5].cpu().numpy().reshape(v_ref.shape), v_ref)
        assert np.array_equal(job[6].cpu().numpy().view(np.uint32).reshape(m_ref.shape), m_ref)
        assert np.array_equal(job[7].cpu().numpy(), s_ref)


def test_staged_units_of_several_warps_and_of_one_in_turn():
    """Rows of four warps, of one and of four again in the consecutive units of every resident block (444 of them): the slots
    of the row maximum are shared by the rows of several warps alone."""
    import paper_2206_15014_b200 as nm
    from gpu_util import DEV, to_dev
    blocks = 3 * torch.cuda.get_device_properties(DEV).multi_processor_count
    jobs, refs = [], []
    for i, k in enumerate([4096, 1024, 4096, 1024, 2048, 4096]):
        out = blocks * 4096 // k  # one unit per block
        W, U = wl.pack_sweep_matrix(31, i, out, k)
        W *= (1.0 + np.arange(out, dtype=np.float32) % 7)[:, None]  # neighbouring rows differ in scale
        vb, mb = nm.nm_packed_sizes(out, k, 2, 4, 8)
        jobs.append((to_dev(W), to_dev(U), 2, 4, 8, torch.zeros(vb, dtype=torch.uint8, device=DEV),
                     torch.zeros(mb // 4, dtype=torch.int32, device=DEV), torch.zeros(out, dtype=torch.float32, device=DEV)))
        refs.append(oracle.project_pack(W, U, 2, 4, 8))
    ws_bytes = nm.nm_pack_workspace_bytes(len(jobs))
    ws = torch.empty(ws_bytes, dtype=torch.uint8, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    nm.nm_debug_set_option("pack_form", 2)
    try:
        for _ in range(5):
            nm.nm_project_pack_batched(nm.make_pack_jobs(jobs), len(jobs), ws, ws_bytes, status)
        assert nm.nm_poll_status(status) == 0
    finally:
        nm.nm_debug_set_option("pack_form", 0)
    for job, (v_ref, m_ref, s_ref) in zip(jobs, refs):
        assert np.array_equal(job[7].cpu().numpy(), s_ref)
        assert np.array_equal(job[5].cpu().numpy().reshape(v_ref.shape), v_ref)
        assert np.array_equal(job[6].cpu().numpy().view(np.uint32).reshape(m_ref.shape), m_ref)


@pytest.mark.parametrize("n,m,bits", [(2, 4, 8), (4, 8, 8), (1, 4, 4), (4, 4, 4)])
def test_forms_admm_step(n, m, bits):
    """Dense outputs (Z, U_next) besides the packed ones (the direct form only)."""
    import paper_2206_15014_b200 as nm
    from gpu_util import DEV, to_dev
    oracle.set_threads(oracle.max_threads())
    for seed, (out, k) in enumerate([(3000, 1024), (301, 4096), (9, 1032)]):
        W, U = wl.pack_sweep_matrix(23, seed, out, k)
        Z = torch.full((out + 1, k), float("nan"), dtype=torch.float32, device=DEV)
        Un = torch.full((out + 1, k), float("nan"), dtype=torch.float32, device=DEV)
        status = torch.zeros(1, dtype=torch.int32, device=DEV)
        vb, mb = nm.nm_packed_sizes(out, k, n, m, bits)
        values = torch.zeros(vb, dtype=torch.uint8, device=DEV)
        meta = torch.zeros(max(mb // 4, 1), dtype=torch.int32, device=DEV)
        scales = torch.zeros(out, dtype=torch.float32, device=DEV)
        nm.nm_admm_project(to_dev(W), to_dev(U), out, k, n, m, bits, Z, Un, values, meta if n != m else None, scales,
                           status=status)
        assert nm.nm_poll_status(status) == 0
        Zh, Uh = Z.cpu().numpy(), Un.cpu().numpy()
        assert np.isnan(Zh[out]).all() and np.isnan(Uh[out]).all(), "written past the last row"
        Zr, Unr, sr = oracle.admm_step(W, U, n, m, bits)
        assert np.array_equal(Zh[:out], Zr) and np.array_equal(Uh[:out], Unr)
        v_ref, meta_ref, s_ref = oracle.project_pack(W, U, n, m, bits)
        assert np.array_equal(scales.cpu().numpy(), s_ref)
        assert np.array_equal(values.cpu().numpy(), np.asarray(v_ref).reshape(-1))
        if n != m:
            assert np.array_equal(meta.cpu().numpy().view(np.uint32)[: mb // 4], np.asarray(meta_ref).reshape(-1))


def _automatic(outs, k, with_u, n=2, m=4, bits=8):
    """The jobs in one call with the library's own choice of form, every output against the oracle."""
    import paper_2206_15014_b200 as nm
    from gpu_util import DEV, to_dev
    oracle.set_threads(oracle.max_threads())
    jobs, refs = [], []
    for i, (out, has_u) in enumerate(zip(outs, with_u)):
        W, U = wl.pack_sweep_matrix(41, i, out, k)
        U = U if has_u else None
        vb, mb = nm.nm_packed_sizes(out, k, n, m, bits)
        jobs.append((to_dev(W), None if U is None else to_dev(U), n, m, bits, torch.zeros(vb, dtype=torch.uint8, device=DEV),
                     torch.zeros(mb // 4, dtype=torch.int32, device=DEV), torch.zeros(out, dtype=torch.float32, device=DEV)))
        refs.append(oracle.project_pack(W, U, n, m, bits))
    ws_bytes = nm.nm_pack_workspace_bytes(len(jobs))
    ws = torch.empty(ws_bytes, dtype=torch.uint8, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    nm.nm_project_pack_batched(nm.make_pack_jobs(jobs), len(jobs), ws, ws_bytes, status)
    assert nm.nm_poll_status(status) == 0
    for job, (v_ref, m_ref, s_ref) in zip(jobs, refs):
        assert np.array_equal(job[7].cpu().numpy(), s_ref)
        assert np.array_equal(job[5].cpu().numpy().reshape(v_ref.shape), v_ref)
        assert np.array_equal(job[6].cpu().numpy().view(np.uint32).reshape(m_ref.shape), m_ref)


@pytest.mark.parametrize("n,m,bits", [(1, 4, 4), (2, 4, 8), (1, 8, 8), (2, 8, 4)])
@pytest.mark.parametrize("blocks_per_sm,beyond", [(5, 0), (5, 1), (8, 0), (8, 1)])
@pytest.mark.parametrize("k", [1024, 3072])
def test_both_sides_of_the_librarys_choice(n, m, bits, blocks_per_sm, beyond, k):
    """One matrix with two operands: up to five blocks a multiprocessor direct with more registers, up to eight direct, beyond
    staged (rows of 3072: 2:4 only)."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rows = 4 if k == 1024 else 1  # a block's
    _automatic([rows * (blocks_per_sm * sms + beyond)], k, [True], n, m, bits)


@pytest.mark.parametrize("beyond", [0, 1])
@pytest.mark.parametrize("n,m", [(2, 4), (1, 8)])
def test_six_rounds_of_several_matrices(n, m, beyond):
    """Two matrices: up to six rounds of eight blocks a multiprocessor staged, beyond direct."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    _automatic([4 * (3 * 8 * sms), 4 * (3 * 8 * sms + beyond)], 1024, [True, True], n, m)


@pytest.mark.parametrize("with_u", [[True, True, True], [True, False, True]])
def test_one_operand_in_a_batch_of_two_operand_jobs(with_u):
    """Three rounds of blocks: staged when every job has a U, direct when one has none."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    _automatic([4 * 8 * sms] * 3, 1024, with_u, bits=4)


def test_few_blocks_of_every_pattern():
    """Launches of a few blocks with two operands, rows of every kind: the direct form with more registers."""
    for n, m in PATTERNS:
        for out, k in ((7, 768), (9, 1032 if m == 4 else 1040), (130, 1024), (3, 4096)):
            if n == m:
                W, U = wl.pack_sweep_matrix(43, out, out, k)
                _check_pack(W, U, n, m, 8)
            else:
                _automatic([out], k, [True], n, m, 8)
