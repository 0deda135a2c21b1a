"""Calls at the edges of what the solver takes: product rows around the length of the SpGEMM
table, aggregates larger than shared memory, empty classes of unknowns, too little device
memory, a hierarchy that changes its shape, meshes of few cells, a device that was reset."""
import contextlib
import os
import subprocess
import sys
import time

import numpy as np
import pytest
import scipy.sparse as sp

import fsigen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_05648_gb300 import build
    build.build()
    return torch


def _system(**blocks):
    """CSR and class offsets of a 2D system: `blocks` names class pairs such as m_m, v_p (classes m, sv, su, v, p);
    a class without a diagonal block is one node of identity rows (one entry for p)."""
    names = ("m", "sv", "su", "v", "p")
    size = {k: (blocks[f"{k}_{k}"].shape[0] if f"{k}_{k}" in blocks else 1 if k == "p" else 2) for k in names}
    grid = [[blocks.get(f"{r}_{c}", sp.identity(size[r]) if r == c else sp.csr_matrix((size[r], size[c])))
             for c in names] for r in names]
    A = sp.block_array(grid, format="csr") if hasattr(sp, "block_array") else sp.bmat(grid, format="csr")
    A.sort_indices()
    return A, np.cumsum([0] + [size[k] for k in names]).astype(np.int64)


def _context(A, off, **params):
    import paper_1801_05648_gb300 as P
    return P.FSISolver(2, A.indptr.astype(np.int64), A.indices.astype(np.int32), A.data.astype(np.float64), off, None,
                       P.default_params(2, **params))


# pressures below and above 16 rows per SM: a block or a warp per product row
@pytest.mark.parametrize("n_p", [900, 2600])
@pytest.mark.parametrize("cols", [767, 768, 769, 900])
def test_product_rows_around_the_table(n_p, cols, torch_cuda):
    """S_p = I - e_0 w^T with w on `cols` pressures: a row of up to 768 columns is taken, and S_p^-1 b is
    b + e_0 (w.b) / (1 - w_0) to the rounding of a well-conditioned inverse; a longer one is refused, and
    the context is good again with the next values."""
    torch = torch_cuda
    import paper_1801_05648_gb300 as P
    w = np.zeros(n_p)
    w[:cols] = 0.5 / cols
    first = np.arange(n_p) * 2
    v_p = sp.csr_matrix((np.ones(n_p), (first, np.arange(n_p))), (2 * n_p, n_p))
    p_v = sp.csr_matrix((w[:cols], (np.zeros(cols, int), first[:cols])), (n_p, 2 * n_p))
    A, off = _system(v_v=sp.identity(2 * n_p), v_p=v_p, p_v=p_v, p_p=sp.identity(n_p))
    S = _context(A, off, coarse_max=8000)
    b = np.random.default_rng(cols).standard_normal(n_p)
    x = torch.empty(n_p, dtype=torch.float64, device="cuda")
    for _ in range(2):
        if cols <= 768:
            S.precond_build("fp64")
            S.apply_block("pressure_schur", torch.tensor(b, device="cuda"), x)
            want = b.copy()
            want[0] += (w @ b) / (1 - w[0])
            assert np.abs(x.cpu().numpy() - want).max() <= 1e-12 * np.abs(b).max()
        else:
            with pytest.raises(P.FSIError) as e:
                S.precond_build("fp64")
            assert e.value.code == P.FSI_EINVAL and "768" in str(e.value)
        S.update_values(torch.tensor(A.data, device="cuda"))
    S.close()


def test_an_aggregate_larger_than_shared_memory(torch_cuda):
    """A star of 1,001 nodes is one aggregate: 4,004 values to orthogonalise, more than the 2,560 that a
    warp keeps in shared memory; and R A has one row of 1,001 columns, which the optional product
    -(R A) does not take.  A V-cycle as the oracle's (sums of 2,002 terms, some ten passes: 1e-10)."""
    torch = torch_cuda
    from oracle import amg
    n = 1001
    S1 = sp.diags(np.concatenate([[1000.0], np.full(n - 1, 1.5)])).tolil()
    S1[0, 1:] = -1.0
    S1[1:, 0] = -1.0
    M = sp.kron(S1.tocsr(), sp.identity(2)).tocsr()
    A, off = _system(m_m=M)
    S = _context(A, off, coarse_max=8, strength_theta=0.01)
    S.precond_build("fp64")
    H = amg.sa_setup(A[: 2 * n, : 2 * n].tocsr(), 2, amg.translations(n, 2),
                     amg.AMGParams(coarse_max=8, theta=0.01))
    assert S.amg_info("mesh")["levels"] == len(H.levels) == 2
    assert H.levels[0].nagg == 1
    b = np.random.default_rng(0).standard_normal(2 * n)
    x = torch.empty(2 * n, dtype=torch.float64, device="cuda")
    S.apply_block("mesh", torch.tensor(b, device="cuda"), x)
    want = amg.vcycle(H, b)
    assert np.linalg.norm(x.cpu().numpy() - want) <= 1e-10 * np.linalg.norm(want)
    S.close()


# the classes of unknowns that are left out, out of m, sv, su, v, p
@pytest.mark.parametrize("empty", [("m",), ("sv", "su"), ("v",), ("p",), ("v", "p"), ("m", "sv", "su", "v"),
                                   ("m", "sv", "su", "p"), ("sv", "su", "v", "p")])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_empty_classes(empty, precision, torch_cuda):
    """A system without one or several classes: the operator is the host's product within its rounding,
    (row length + 2) u |A| |x|, into a vector that held something else, and the solution has a
    residual of 1e-10."""
    torch = torch_cuda
    rng = np.random.default_rng(7)
    size = {k: 0 if k in empty else 30 if k == "p" else 60 for k in ("m", "sv", "su", "v", "p")}
    n = sum(size.values())
    A = sp.random(n, n, 0.1, random_state=rng, data_rvs=rng.standard_normal).tocsr()
    A = (A + sp.identity(n) * 20.0).tocsr()
    A.sort_indices()
    off = np.cumsum([0] + list(size.values())).astype(np.int64)
    S = _context(A, off, maxit=300)
    x = rng.standard_normal(n)
    y = torch.full((n,), 7.0, dtype=torch.float64, device="cuda")
    S.apply_operator(torch.tensor(x, device="cuda"), y)
    bound = (np.diff(A.indptr) + 2) * np.finfo(float).eps * (abs(A) @ np.abs(x))
    assert (np.abs(y.cpu().numpy() - A @ x) <= bound).all()
    S.precond_build(precision)
    b = A @ x
    z = torch.full((n,), 7.0, dtype=torch.float64, device="cuda")
    st = S.solve(torch.tensor(b, device="cuda"), z, 1e-10)
    assert st.status == 0 and np.linalg.norm(b - A @ z.cpu().numpy()) <= 1.001e-10 * np.linalg.norm(b)
    S.close()


@contextlib.contextmanager
def _memory_left(torch, nbytes):
    """The device with about nbytes free while the block runs."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    ballast = []
    for size in (32 << 30, 4 << 30, 512 << 20, 64 << 20, 8 << 20, 2 << 20):
        while torch.cuda.mem_get_info()[0] >= nbytes + size:
            try:
                ballast.append(torch.empty(size, dtype=torch.uint8, device="cuda"))
            except torch.OutOfMemoryError:
                break
    try:
        yield
    finally:
        torch.cuda.synchronize()
        del ballast
        torch.cuda.empty_cache()


def test_training_step_after_a_failed_allocation(torch_cuda):
    """A training step that does not get its memory says so, and the next one, with memory, has the loss and the
    gradient of a trainer that never failed."""
    torch = torch_cuda
    import paper_1801_05648_gb300 as P
    pb = fsigen.get_problem(fsigen.CONFIGS["2d_tiny"].with_(name="t", n=(96, 64)))
    U = pb.seeded_state(0, 5e-3)
    S = P.FSISolver(pb.dim, pb.rowptr, pb.colind, pb.jacobian(U, U), pb.offsets, pb.solid_node_coords(),
                    P.default_params(2))
    S.learned_setup(*pb.node_map())
    r = torch.tensor(np.random.default_rng(1).standard_normal(pb.n), device="cuda")
    ref = P.Trainer(seed=3)
    loss = ref.step(S, r)
    grad = ref.get()[2]
    failed = 0
    for mb in (1, 6, 12, 24, 40):
        T = P.Trainer(seed=3)
        with _memory_left(torch, mb << 20):
            try:
                T.step(S, r)
            except P.FSIError as e:
                assert e.code == P.FSI_ENOMEM
                failed += 1
            else:
                continue
        assert T.step(S, r) == loss and np.array_equal(T.get()[2], grad)
        T.close()
    assert failed >= 2
    S.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_build_after_a_failed_allocation(precision, torch_cuda):
    """A build that runs out of memory, at whatever point, says so; the same call with memory builds what a
    context that never failed has."""
    torch = torch_cuda
    import paper_1801_05648_gb300 as P
    pb = fsigen.get_problem(fsigen.CONFIGS["2d_tiny"].with_(name="b", n=(128, 96)))
    U = pb.seeded_state(0, 5e-3)
    vals = torch.tensor(pb.jacobian(U, U), device="cuda")
    r = torch.tensor(np.random.default_rng(2).standard_normal(pb.n), device="cuda")

    def context():
        S = P.FSISolver(pb.dim, pb.rowptr, pb.colind, None, pb.offsets, pb.solid_node_coords(), P.default_params(2))
        S.update_values(vals)
        return S

    def applied(S):
        z = torch.empty_like(r)
        S.apply_block("precond", r, z)
        return z
    S = context()
    S.precond_build(precision)
    want = applied(S)
    S.close()
    failed = 0
    for mb in (0, 40, 80, 120, 160, 200, 240, 280, 320, 400, 480):
        S = context()
        with _memory_left(torch, mb << 20):
            try:
                S.precond_build(precision)
            except P.FSIError as e:
                assert e.code == P.FSI_ENOMEM, e
                failed += 1
            else:
                S.close()
                break
        S.precond_build(precision)
        assert torch.equal(applied(S), want)
        S.update_values(vals)
        S.precond_build(precision)
        assert torch.equal(applied(S), want)
        S.close()
    assert failed >= 3


# meshes where the FP32 restriction's form changes with 2 bytes more or less per block of level 0
@pytest.mark.parametrize("cells", [(32, 30), (30, 30), (48, 31)])
def test_rebuild_equals_a_fresh_context(cells, torch_cuda):
    """A second FP32 build of the same values has the bits of the first."""
    torch = torch_cuda
    import paper_1801_05648_gb300 as P
    pb = fsigen.get_problem(fsigen.FSIConfig("c", 2, cells))
    U = pb.seeded_state(0, 5e-3)
    vals = torch.tensor(pb.jacobian(U, U), device="cuda")
    r = torch.tensor(np.random.default_rng(2).standard_normal(pb.n), device="cuda")
    S = P.FSISolver(pb.dim, pb.rowptr, pb.colind, None, pb.offsets, pb.solid_node_coords(), P.default_params(2))
    z = [torch.empty_like(r) for _ in range(3)]
    for k in range(3):
        S.update_values(vals)
        S.precond_build("fp32")
        S.apply_block("precond", r, z[k])
    assert torch.equal(z[0], z[1]) and torch.equal(z[0], z[2])
    S.close()


def test_a_build_releases_the_blocks_it_used_up(torch_cuda):
    """After a build the solid's velocity block lives on in S_hat alone: new values take its memory again
    (memory is compared with the pools emptied, which a failed allocation does)."""
    torch = torch_cuda
    import paper_1801_05648_gb300 as P
    pb = fsigen.get_problem(fsigen.CONFIGS["2d_tiny"].with_(name="b", n=(256, 128)))
    U = pb.seeded_state(0, 5e-3)
    vals = torch.tensor(pb.jacobian(U, U), device="cuda")
    S = P.FSISolver(pb.dim, pb.rowptr, pb.colind, None, pb.offsets, pb.solid_node_coords(), P.default_params(2))

    def free():
        with _memory_left(torch, 1 << 20):
            with contextlib.suppress(P.FSIError):
                P.FSIAssembler.from_problem(pb).close()
        return torch.cuda.mem_get_info()[0]
    o = pb.offsets
    rows = slice(int(pb.rowptr[o[1]]), int(pb.rowptr[o[2]]))
    cols = pb.colind[rows]
    avv = 8 * int(((cols >= o[1]) & (cols < o[2])).sum())
    assert avv > 8 << 20
    S.update_values(vals)
    S.precond_build("fp64")
    built = free()
    S.update_values(vals)
    assert built - free() >= avv - (4 << 20)                # whole driver pages of 2 MB
    S.close()


def _anisotropic_grid(n, wy):
    """Five-point operator on n x n nodes, coupling -1 in x and -wy in y, two components."""
    T = sp.diags([-np.ones(n - 1), -np.ones(n - 1)], [-1, 1])
    K = sp.kron(sp.identity(n), T) + wy * sp.kron(T, sp.identity(n))
    K = K + sp.diags(np.asarray(-K.sum(1)).ravel() + 0.1)
    return sp.kron(K, sp.identity(2)).tocsr()


@pytest.mark.parametrize("flag", ["FSI_GRID_COARSE", "FSI_CLUSTER_COARSE"])
def test_coarse_launch_follows_the_hierarchy(flag, torch_cuda):
    """Values whose first coarse level is small enough for the single coarse launch, then values whose is not
    (coarsened along x alone), then the first again: each build as the oracle's V-cycle."""
    torch = torch_cuda
    import paper_1801_05648_gb300 as P
    from oracle import amg
    values = [_anisotropic_grid(40, w) for w in (1.0, 1e-4)]
    assert np.array_equal(values[0].indices, values[1].indices)
    H = [amg.sa_setup(M, 2, amg.translations(1600, 2), amg.AMGParams(coarse_max=300)) for M in values]
    limit = 1e5                                             # bytes of a level's FP64 values
    size = [[sp.bsr_matrix(h.levels[k].A, blocksize=(2, 2)).indices.size * 32 for h in H] for k in (0, 1)]
    assert [len(h.levels) for h in H] == [3, 3] and size[1][0] < limit < size[1][1] < size[0][0]
    A, off = _system(m_m=values[0])
    S = _context(A, off, coarse_max=300, cluster_max_bytes=limit, flags=getattr(P, flag))
    b = np.random.default_rng(0).standard_normal(3200)
    x = torch.empty(3200, dtype=torch.float64, device="cuda")
    for k in (0, 1, 0):
        data = A.copy()
        data.data[: values[k].nnz] = values[k].data
        S.update_values(torch.tensor(data.data, device="cuda"))
        S.precond_build("fp64")
        S.apply_block("mesh", torch.tensor(b, device="cuda"), x)
        want = amg.vcycle(H[k], b)
        assert np.linalg.norm(x.cpu().numpy() - want) <= 1e-10 * np.linalg.norm(want)
    S.check_device_errors()
    S.close()


# cells per colour that give a CTA 1, 2, 3, 8 (Jacobian) and 1, 2, 3, 9, 28 (residual) cells, the last CTA fewer
@pytest.mark.parametrize("cells", [(34, 35), (38, 37), (50, 49), (101, 99), (190, 188), (14, 15, 13)])
def test_assembly_of_groups_of_cells(cells, torch_cuda):
    """Entries within 1e-12 of the row's largest magnitude of the host assembly's, however many cells a CTA takes."""
    torch = torch_cuda
    import paper_1801_05648_gb300 as P
    pb = fsigen.get_problem(fsigen.FSIConfig("a", len(cells), cells, theta=0.5))
    U = pb.seeded_state(4, 5e-3)
    asm = P.FSIAssembler.from_problem(pb)
    u, uo = torch.tensor(U, device="cuda"), torch.tensor(0.9 * U, device="cuda")
    R, J = torch.empty_like(u), torch.empty(pb.nnz, dtype=torch.float64, device="cuda")
    asm.residual(u, uo, R)
    asm.jacobian(u, uo, J)
    Rh, Jh = pb.residual(U, 0.9 * U), pb.jacobian(U, 0.9 * U)
    assert np.abs(R.cpu().numpy() - Rh).max() <= 1e-12 * np.abs(Rh).max()
    big = np.maximum.reduceat(np.abs(Jh), pb.rowptr[:-1])
    assert np.max(np.abs(J.cpu().numpy() - Jh) / np.repeat(big, np.diff(pb.rowptr))) <= 1e-12
    asm.close()


def test_assembly_of_a_small_mesh_is_spread_over_the_gpu(torch_cuda):
    """98 cells, a fortieth of the work of 90x45 and less than a hundredth of 180x90's, take less than four fifths
    of their time (launches and host work are in both; in groups of the size that suits large meshes the
    Jacobian of the small mesh took as long as the one of 90x45, its residual 0.9 of 180x90's)."""
    torch = torch_cuda
    import paper_1801_05648_gb300 as P

    def median(cells, call):
        pb = fsigen.get_problem(fsigen.FSIConfig("a", 2, cells))
        u = torch.tensor(pb.seeded_state(4, 5e-3), device="cuda")
        out = torch.empty(pb.nnz if call == "jacobian" else pb.n, dtype=torch.float64, device="cuda")
        asm = P.FSIAssembler.from_problem(pb)
        run = getattr(asm, call)
        times = []
        for _ in range(40):
            torch.cuda.synchronize()
            t = time.perf_counter()
            run(u, u, out)
            times.append(time.perf_counter() - t)
        asm.close()
        return sorted(times[10:])[15]
    for call, cells in (("jacobian", (90, 45)), ("residual", (180, 90))):
        small, large = median((14, 7), call), median(cells, call)
        assert small < 0.8 * large, (call, small, large)


# Everything a Newton correction calls, on the library alone (a process's PyTorch does not outlive a reset).
_RESET = r"""
import ctypes
import numpy as np
import fsigen
import paper_1801_05648_gb300.fsi as F

lib = F.load_library()
cudart = ctypes.CDLL("libcudart.so.13")
cudart.cudaMalloc.argtypes = [ctypes.POINTER(ctypes.c_void_p), ctypes.c_size_t]
cudart.cudaMemcpy.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int]
pb = fsigen.get_problem(fsigen.FSIConfig("c", 2, (64, 48)))
U = pb.seeded_state(0, 5e-3)
rng = np.random.default_rng(0)
b = rng.standard_normal(pb.n)
bits = (rng.standard_normal(F.mlp_params(2)).astype(np.float32) * 0.1).view(np.uint32) >> 16
bits = np.ascontiguousarray(bits, np.uint16)


def ok(rc):
    assert rc == 0, rc


def dev(a):
    p = ctypes.c_void_p()
    ok(cudart.cudaMalloc(ctypes.byref(p), a.nbytes))
    ok(cudart.cudaMemcpy(p, a.ctypes.data, a.nbytes, 1))
    return p


def host(p, n):
    a = np.empty(n)
    ok(cudart.cudaDeviceSynchronize())
    ok(cudart.cudaMemcpy(a.ctypes.data, p, a.nbytes, 2))
    return a


def ptr(a, t):
    return a.ctypes.data_as(ctypes.POINTER(t))


def correction():
    cd, cf = pb.cell_map()
    cfg, m = pb.cfg, F.AsmMesh()
    arrays = [np.ascontiguousarray(cd, np.int32), np.ascontiguousarray(cf, np.uint32),
              np.ascontiguousarray(pb.rowptr, np.int64), np.ascontiguousarray(pb.colind, np.int32),
              np.ascontiguousarray(pb.fixed, np.uint8), np.ascontiguousarray(pb.offsets, np.int64)]
    m.dim, m.pressure, m.n = 2, 0, pb.n
    for d in range(3):
        m.cells[d], m.h[d] = (cfg.n[d], cfg.L[d] / cfg.n[d]) if d < 2 else (1, 1.0)
    m.cell_dof, m.cell_flags = ptr(arrays[0], ctypes.c_int32), ptr(arrays[1], ctypes.c_uint32)
    m.rowptr, m.colind, m.row_fixed = ptr(arrays[2], ctypes.c_int64), ptr(arrays[3], ctypes.c_int32), ptr(arrays[4], ctypes.c_uint8)
    ph = F.AsmPhysics(**{k: float(getattr(cfg, k)) for k in ("rho_f", "nu_f", "mu_s", "lambda_s", "rho_s", "dt", "theta")})
    asm, ctx = ctypes.c_void_p(), ctypes.c_void_p()
    u, vals, r, z, x = dev(U), dev(np.zeros(pb.nnz)), dev(b), dev(np.zeros(pb.n)), dev(np.zeros(pb.n))
    ok(lib.fsi_asm_create(ctypes.byref(asm), ctypes.byref(m), ctypes.byref(ph), None))
    ok(lib.fsi_asm_residual(asm, u, u, z, None, None))
    out = [host(z, pb.n)]
    ok(lib.fsi_asm_jacobian(asm, u, u, vals, None))
    prm = F.default_params(2)
    prm.flags = F.FSI_USE_GRAPHS
    ok(lib.fsi_setup(ctypes.byref(ctx), 2, pb.n, ptr(arrays[2], ctypes.c_int64), ptr(arrays[3], ctypes.c_int32), None,
                     ptr(arrays[5], ctypes.c_int64), None, ctypes.byref(prm), None))
    ok(lib.fsi_update_values(ctx, vals))
    ok(lib.fsi_precond_build(ctx, 1, None))
    ok(lib.fsi_apply_block(ctx, 7, r, z))
    out.append(host(z, pb.n))
    st = F.Stats()
    ok(lib.fsi_solve(ctx, r, x, 1e-8, ctypes.byref(st)))
    out.append(host(x, pb.n))
    nd, pt = (np.ascontiguousarray(a, np.int32) for a in pb.node_map())
    one = np.ones(5, np.float32)
    ok(lib.fsi_learned_setup(ctx, len(nd), ptr(nd, ctypes.c_int32), ptr(pt, ctypes.c_int32)))
    ok(lib.fsi_learned_set_weights(ctx, ptr(one, ctypes.c_float), ptr(one, ctypes.c_float), ptr(bits, ctypes.c_uint16)))
    ok(lib.fsi_learned_apply(ctx, r, z))
    out.append(host(z, pb.n))
    lib.fsi_free(ctx)
    lib.fsi_asm_free(asm)
    return out


first = correction()
ok(cudart.cudaDeviceReset())
second = correction()
assert all(np.array_equal(a, c) and np.abs(a).max() > 0 for a, c in zip(first, second))
print("same")
"""


def test_contexts_after_a_device_reset(torch_cuda):
    """What is set up once per device (streams, kernels' attributes) is set up again for contexts made after a
    reset of the device: same bits."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _RESET], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "same" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
