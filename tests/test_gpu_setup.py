"""Set-up kernels at the sizes where they can go wrong: the panelled dense inverse of the
coarsest level around its panel, tile and cluster sizes (with pivoting), preconditioner
rebuilds that reuse a context's memory, builds in several threads, and the device
assembly on meshes smaller than its cell groups and on patterns that lack entries; and the
solver's launches that overlap or are left out (queued products, the second Gram-Schmidt pass)."""
import threading

import numpy as np
import pytest

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


def _dense_system(n, seed):
    """A CSR whose mesh block is a dense random n x n matrix (no diagonal dominance) and
    one identity node in each other class."""
    rng = np.random.default_rng(seed)
    A = rng.standard_normal((n, n))
    m = n + 7
    rowptr = np.concatenate([np.arange(n + 1) * n, n * n + 1 + np.arange(7)]).astype(np.int64)
    colind = np.concatenate([np.tile(np.arange(n), n), np.arange(n, m)]).astype(np.int32)
    vals = np.concatenate([A.ravel(), np.ones(7)])
    return A, rowptr, colind, vals, np.array([0, n, n + 2, n + 4, n + 6, n + 7], np.int64)


@pytest.mark.parametrize("n", [2, 14, 16, 18, 32, 34, 254, 256, 258, 510, 514, 1022, 1026])
def test_dense_inverse_sizes(n, torch_cuda):
    """Partial pivoting keeps the backward error of the inverse's columns near n u growth;
    100 n u max|A^-1| max|A| leaves room for the growth of random matrices (about n^(2/3))."""
    torch = torch_cuda
    import paper_1801_05648_gb300 as P
    A, rowptr, colind, vals, off = _dense_system(n, n)
    S = P.FSISolver(2, rowptr, colind, vals, off, None, P.default_params(2))
    S.precond_build("fp64")
    assert S.amg_info("mesh")["levels"] == 1
    b = np.random.default_rng(1).standard_normal(n)
    x = torch.empty(n, dtype=torch.float64, device="cuda")
    S.apply_block("mesh", torch.tensor(b, device="cuda"), x)
    want = np.linalg.solve(A, b)
    inv = np.linalg.inv(A)
    bound = 100 * n * np.finfo(float).eps * np.abs(inv).max() * np.abs(A).max() * np.abs(want).max()
    assert np.abs(x.cpu().numpy() - want).max() <= bound
    S.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_rebuilds_equal_fresh_contexts(precision, torch_cuda):
    """Two sets of values in turn through one context: every rebuild gives the bits of a new context."""
    torch = torch_cuda
    import paper_1801_05648_gb300 as P
    cfg = fsigen.CONFIGS["2d_tiny"].with_(name="r", n=(37, 19))
    pb = fsigen.get_problem(cfg)
    vals = []
    for seed in (0, 1):
        U = pb.seeded_state(seed, 5e-3)
        vals.append(torch.tensor(pb.jacobian(U, U), device="cuda"))
    r = torch.tensor(np.random.default_rng(2).standard_normal(pb.n), device="cuda")

    def solver():
        return P.FSISolver(pb.dim, pb.rowptr, pb.colind, None, pb.offsets, pb.solid_node_coords(),
                           P.default_params(2))

    def apply(S, v):
        z = torch.empty_like(r)
        S.update_values(v)
        S.precond_build(precision)
        S.apply_block("precond", r, z)
        return z
    fresh = [apply(solver(), v) for v in vals]
    assert not torch.equal(fresh[0], fresh[1])
    S = solver()
    for k in (0, 1, 0, 0, 1):
        assert torch.equal(apply(S, vals[k]), fresh[k])
    # several contexts built at the same time by several threads
    got = [None] * 4

    def work(i):
        got[i] = apply(solver(), vals[i % 2])
    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for i in range(4):
        assert torch.equal(got[i], fresh[i % 2])


def test_failed_build_leaves_a_usable_error(torch_cuda):
    """A coarsest level too large for the dense inverse is refused, and refused again until the
    context gets new values."""
    torch = torch_cuda
    import paper_1801_05648_gb300 as P
    pb = fsigen.get_problem(fsigen.CONFIGS["2d_tiny"].with_(name="f", n=(64, 64)))
    U = pb.seeded_state(0, 5e-3)
    v = torch.tensor(pb.jacobian(U, U), device="cuda")
    S = P.FSISolver(pb.dim, pb.rowptr, pb.colind, None, pb.offsets, pb.solid_node_coords(),
                    P.default_params(2, max_levels=1))
    for _ in range(2):
        S.update_values(v)
        with pytest.raises(P.FSIError) as e:
            S.precond_build("fp32")
        assert e.value.code == P.FSI_EINVAL
        with pytest.raises(P.FSIError):
            S.precond_build("fp32")
    S.close()


def _assembled(torch, P, pb, U, Uold, rowptr, colind):
    cfg = pb.cfg
    cd, cf = pb.cell_map()
    phys = dict(rho_f=cfg.rho_f, nu_f=cfg.nu_f, mu_s=cfg.mu_s, lambda_s=cfg.lambda_s, rho_s=cfg.rho_s, dt=cfg.dt,
                theta=cfg.theta)
    asm = P.FSIAssembler(pb.dim, cfg.n, [cfg.L[d] / cfg.n[d] for d in range(pb.dim)], pb.n, cd, cf, rowptr, colind,
                         pb.fixed, phys, pressure=cfg.pressure)
    Ud, Uo = torch.tensor(U, device="cuda"), torch.tensor(Uold, device="cuda")
    R = torch.empty_like(Ud)
    vals = torch.empty(len(colind), dtype=torch.float64, device="cuda")
    mj = asm.residual(Ud, Uo, R)
    assert asm.jacobian(Ud, Uo, vals) == mj[0]
    return R.cpu().numpy(), vals.cpu().numpy(), mj


# cells per colour below, at and above the groups of 8 (Jacobian) and 28 (residual) cells
@pytest.mark.parametrize("cells", [(3, 3), (7, 5), (8, 7), (9, 9), (15, 15), (3, 4, 3), (5, 4, 4)])
@pytest.mark.parametrize("pressure", ["q1", "p1disc"])
def test_assembly_of_small_meshes(cells, pressure, torch_cuda):
    """Entries within 1e-12 of the row's largest magnitude of the host assembly's."""
    import paper_1801_05648_gb300 as P
    cfg = fsigen.FSIConfig("a", len(cells), cells, theta=0.5, pressure=pressure)
    pb = fsigen.get_problem(cfg)
    U = pb.seeded_state(4, 5e-3)
    R, vals, (mj, rmax) = _assembled(torch_cuda, P, pb, U, 0.9 * U, pb.rowptr, pb.colind)
    Rh, Jh = pb.residual(U, 0.9 * U), pb.jacobian(U, 0.9 * U)
    assert np.abs(R - Rh).max() <= 1e-12 * np.abs(Rh).max()
    assert rmax == np.abs(R).max()
    assert mj == pytest.approx(pb.min_J, rel=1e-14)
    rows = np.repeat(np.arange(pb.n), np.diff(pb.rowptr))
    big = np.zeros(pb.n)
    np.maximum.at(big, rows, np.abs(Jh))
    assert np.max(np.abs(vals - Jh) / big[rows]) <= 1e-12


@pytest.mark.parametrize("cells", [(9, 8), (4, 4, 4)])
def test_assembly_on_patterns_without_the_zero_couplings(cells, torch_cuda):
    """A pattern without the couplings between different components in the solid's kinematic rows
    (zero for every state): the rows of a node's components then differ, so that entries are
    placed one by one.  A pattern that lacks a coupling that is not zero is refused."""
    import paper_1801_05648_gb300 as P
    cfg = fsigen.FSIConfig("a", len(cells), cells)
    pb = fsigen.get_problem(cfg)
    d = pb.dim
    U = pb.seeded_state(4, 5e-3)
    Jh = pb.jacobian(U, U)
    rows = np.repeat(np.arange(pb.n), np.diff(pb.rowptr))
    su = (rows >= pb.offsets[2]) & (rows < pb.offsets[3])
    keep = ~(su & (rows % d != pb.colind % d))        # class offsets are multiples of d
    assert np.all(pb.offsets[:4] % d == 0) and np.all(Jh[~keep] == 0.0) and (~keep).any()
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(rows[keep], minlength=pb.n))])
    _, vals, _ = _assembled(torch_cuda, P, pb, U, U, rowptr, pb.colind[keep])
    big = np.zeros(pb.n)
    np.maximum.at(big, rows, np.abs(Jh))
    assert np.max(np.abs(vals - Jh[keep]) / big[rows[keep]]) <= 1e-12
    gone = np.flatnonzero(keep & (rows != pb.colind) & (np.abs(Jh) > 0.1 * big[rows]) & ~pb.fixed[rows])[0]
    keep[gone] = False
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(rows[keep], minlength=pb.n))])
    with pytest.raises(P.FSIError):
        _assembled(torch_cuda, P, pb, U, U, rowptr, pb.colind[keep])


@pytest.mark.parametrize("graphs", [False, True])
def test_second_gram_schmidt_pass(graphs, torch_cuda):
    """A system whose preconditioned operator is 2/3 I on the right-hand side's space: the Arnoldi defect
    v - A z = v / 3 is parallel to v, the first pass cancels it to rounding, and the step asks
    for its second pass; the first iterate is the solution (10 u for a handful of roundings)."""
    torch = torch_cuda
    import paper_1801_05648_gb300 as P
    off = np.array([0, 2, 6, 10, 12, 13], np.int64)
    rows = [[i] if not 2 <= i < 6 else [i, i + 4] for i in range(13)]      # A_vv = A_vu = I
    rowptr = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    colind = np.concatenate(rows).astype(np.int32)
    S = P.FSISolver(2, rowptr, colind, np.ones(len(colind)), off, None,
                    P.default_params(2, dt_theta=0.5, flags=P.FSI_USE_GRAPHS if graphs else 0))
    S.precond_build("fp64")
    b = np.zeros(13)
    b[2:6] = np.random.default_rng(0).standard_normal(4)
    x = torch.zeros(13, dtype=torch.float64, device="cuda")
    for _ in range(2):
        st = S.solve(torch.tensor(b, device="cuda"), x, 1e-10)
        assert (st.iters, st.reorth_passes) == (1, 1)
        assert np.abs(x.cpu().numpy() - b).max() <= 10 * np.finfo(float).eps * np.abs(b).max()
    S.close()


@pytest.mark.parametrize("cells,precision", [((3, 3), "fp32"), ((16, 16), "fp64"), ((16, 16), "fp32"), ((37, 19), "fp32"),
                                             ((64, 48), "fp32"), ((4, 4, 4), "fp32"), ((7, 5, 6), "fp64")])
def test_queued_products_read_finished_inputs(cells, precision, torch_cuda):
    """Products queued one behind the other, each reading the last one's result, with launches that load
    their matrix before the previous kernel has finished (small levels, and operators on both sides of the
    size where that ends): the bits of the same products with a wait after each, and of a context without overlapped
    launches; and the operator within its rounding, (row length + 2) u |A| |x|, of the host's product."""
    torch = torch_cuda
    import paper_1801_05648_gb300 as P
    from scipy.sparse import csr_matrix
    base = fsigen.CONFIGS["2d_tiny" if len(cells) == 2 else "3d"]
    pb = fsigen.get_problem(base.with_(name="q", n=cells))
    U = pb.seeded_state(0, 5e-3)
    vals = pb.jacobian(U, U)
    x0 = torch.tensor(np.random.default_rng(3).standard_normal(pb.n), device="cuda")

    def chain(flags, sync):
        S = P.FSISolver(pb.dim, pb.rowptr, pb.colind, vals, pb.offsets, pb.solid_node_coords(),
                        P.default_params(pb.dim, flags=flags))
        S.precond_build(precision)
        v = [x0] + [torch.empty_like(x0) for _ in range(12)]
        torch.cuda.synchronize()
        for k in range(0, 12, 2):
            S.apply_operator(v[k], v[k + 1], sync=sync)
            S.apply_block("precond", v[k + 1], v[k + 2], sync=sync)
        torch.cuda.synchronize()
        S.close()
        return v[1:]
    want = chain(P.FSI_NO_PDL, True)
    for sync in (True, False, False):
        assert all(torch.equal(a, b) for a, b in zip(chain(0, sync), want))
    A = csr_matrix((vals, pb.colind, pb.rowptr))
    x = x0.cpu().numpy()
    bound = (np.diff(pb.rowptr) + 2) * np.finfo(float).eps * (abs(A) @ np.abs(x))
    assert (np.abs(want[0].cpu().numpy() - A @ x) <= bound).all()
