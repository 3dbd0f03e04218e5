"""Kernel variants chosen by size, at the sizes where each can go wrong."""
import numpy as np
import pytest

from synth import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_1910_01011_gb300 import api as a
    return a


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def test_short_chunks_fall_back_under_a_budget(api):
    """Where the budget does not hold the partials of short source chunks, the
    FP32 product takes the longer ones: the same bits as with that chunk
    length asked for (640 tiles: four chunks of 160)."""
    s = scenes.sphere_scene(5)
    x = scenes.smooth_trace_vector(s, 3)
    c = api.Context.from_scene(s)
    c.apply(x, precision=api.FP32)
    used = c.memory()[0]
    c.close()
    c = api.Context.from_scene(s, chunk_tiles=160)
    ref = c.apply(x, precision=api.FP32)
    c.close()
    c = api.Context.from_scene(s, hbm_budget_bytes=used - (1 << 20))  # the short chunks' partials miss by 1 MiB
    y = c.apply(x, precision=api.FP32)
    assert np.array_equal(y, ref)
    assert c.memory()[0] < used - (1 << 28)
    c.close()


@pytest.mark.parametrize("m,k,n", [(1, 1, 1), (128, 32, 16), (129, 33, 3), (130, 2049, 16), (19500, 40, 2), (257, 8200, 1),
                                   (640, 300, 17), (384, 513, 64), (150, 290, 65)])
def test_gemm_split_over_ctas(m, k, n):
    """The split-BF16 product with its units spread over the CTAs (up to 64
    right-hand sides) and with whole tiles (more), at ragged sizes; each of the
    k terms is good to ~2^-23, and rounding of FP32 sums grows like sqrt(k)."""
    import torch
    from paper_1910_01011_gb300 import _lib
    from paper_1910_01011_gb300.api import Context
    g = torch.Generator().manual_seed(m + k + n)
    A = torch.randn(m, k, 2, generator=g)
    X = torch.randn(n, k, 2, generator=g)
    Ac, Xc = torch.view_as_complex(A), torch.view_as_complex(X)
    ref = Xc.to(torch.complex128) @ Ac.to(torch.complex128).T
    c = Context(0, hbm_budget_bytes=0)
    d, x, y = Ac.cuda(), Xc.cuda(), torch.full((n, m), float("nan"), dtype=torch.complex64, device="cuda")
    rc = c.lib.bem_zgemm_bf16x3(c.h, m, k, n, d.data_ptr(), x.data_ptr(), y.data_ptr())
    _lib.check(rc, c.h)
    err = (y.cpu().to(torch.complex128) - ref).norm() / ref.norm()
    c.close()
    assert err < 2e-6


@pytest.mark.parametrize("n_gauss", [2, 5, 6, 9])
@pytest.mark.parametrize("name", ["shell", "two"])
def test_near_groups_match_native_fp64(api, name, n_gauss):
    """The double-float near build (rules as groups of points along a line)
    against the native FP64 one over points, for Gauss orders with other group
    counts than the default; double-float evaluations carry ~1e-13."""
    s = scenes.shell_scene(1) if name == "shell" else scenes.two_sphere_scene(1)
    x = scenes.smooth_trace_vector(s, 5)
    y = []
    for native in (0, 1):
        c = api.Context.from_scene(s, n_gauss_singular=n_gauss, fp64_far=native)
        y.append(c.apply(x, precision=api.FP64))
        c.close()
    assert rel(y[0], y[1]) < 1e-12


@pytest.mark.parametrize("name,R", [("sphere", 1), ("sphere", 8), ("two", 9), ("two", 16), ("shell", 17), ("shell", 33)])
def test_fp64_assembled_digits(api, name, R):
    """The assembled FP64 product in fixed-point digits, by its own columns
    (unit vectors, whose digits are exact): vectors of very different sizes,
    with the psi and phi blocks a factor |k| apart, a zero vector, and an
    infinite one that leaves the others alone.  Digits keep 2^-54 of the largest
    scaled entry of a row and of a vector; rows here range over less than 2^12."""
    s = {"sphere": lambda: scenes.sphere_scene(1), "two": lambda: scenes.two_sphere_scene(2),
         "shell": lambda: scenes.shell_scene(1)}[name]()
    c = api.Context.from_scene(s)
    N = c.n_dofs
    A = c.apply(np.eye(N, dtype=np.complex128), precision=api.FP64_ASSEMBLED).T
    rng = np.random.default_rng(R)
    X = np.stack([scenes.smooth_trace_vector(s, r) for r in range(R)]) * 10.0 ** rng.uniform(-150, 150, (R, 1))
    if R > 8:
        X[3] = 0.0
        X[5, N // 2] = np.inf
    Y = c.apply(X if R > 1 else X[0], precision=api.FP64_ASSEMBLED).reshape(R, N)
    c.close()
    for r in range(R):
        if R > 8 and r == 3:
            assert not Y[r].any()
        elif R > 8 and r == 5:
            assert np.isnan(Y[r].real).all()
        else:
            assert rel(Y[r], A @ X[r]) < 1e-12


@pytest.mark.parametrize("name,R", [("ribs", 2), ("kidney", 5), ("lossy", 3), ("phase", 8)])
def test_tensor_core_far_field(api, name, R):
    """Several right-hand sides on meshes large enough for the tensor-core far
    field (at least 96 tiles; target blocks of 128 points straddle tiles and
    domains, a short last group and block, attenuating interior and exterior,
    phases over hundreds of radians), against the FP64 path at the FP32 bar;
    vectors of very different sizes and a zero one."""
    s = {"ribs": lambda: scenes.rib_scene(h=9e-3, freq=0.03e6), "kidney": lambda: scenes.kidney_scene(h=7.5e-3, freq=0.04e6),
         "lossy": lambda: scenes.sphere_scene(4, k0=6.0 + 0.4j, k1=6.5 + 1.5j),
         "phase": lambda: scenes.sphere_scene(4, k0=150.0, k1=160.0 + 0.5j)}[name]()
    c = api.Context.from_scene(s)
    X = np.stack([scenes.smooth_trace_vector(s, r) * 10.0 ** (6 * r - 9) for r in range(R)])
    if R == 5:
        X[3] = 0.0
    Y = c.apply(X, precision=api.FP32)
    Z = c.apply(X, precision=api.FP64)
    for r in range(R):
        if R == 5 and r == 3:
            assert not Y[r].any()
        else:
            assert rel(Y[r], Z[r]) < 2e-5, r
    c.close()


def test_tensor_core_far_field_gives_its_memory_back(api):
    """Under a budget that does not hold the operands next to the rest, the
    product takes the FP32 kernel for all pairs, with the same result to FP32
    accuracy; operands already held go when another allocation needs the room."""
    s = scenes.sphere_scene(4)
    X = np.stack([scenes.smooth_trace_vector(s, r) for r in range(16)])
    c = api.Context.from_scene(s)
    ref = c.apply(X, precision=api.FP32)
    used = c.memory()[0]
    c.close()
    c = api.Context.from_scene(s, hbm_budget_bytes=used - (1 << 22))
    y = c.apply(X, precision=api.FP32)
    assert c.memory()[0] <= used - (1 << 22)
    assert rel(y, ref) < 1e-5
    c.close()
    c = api.Context.from_scene(s, hbm_budget_bytes=used + (16 << 20))  # (host vectors are staged)
    y = c.apply(X, precision=api.FP32)
    assert np.array_equal(y, ref)
    c.apply(X[:8], precision=api.FP64)  # its vectors and partials do not fit beside the operands
    y = c.apply(X[:3], precision=api.FP32)
    assert rel(y, ref[:3]) < 1e-5
    c.close()


@pytest.mark.parametrize("level,R,solver", [(3, 1, 0), (3, 12, 0), (4, 1, 0), (4, 5, 0), (4, 12, 0), (4, 12, 1)])
def test_loose_solves_in_shared_memory(api, level, R, solver):
    """The preconditioner's FP32 solves with a system's vectors in one CTA's
    shared memory (642 and 2,562 vertices: two and eight rows per thread, one
    and two systems per CTA) inside block GMRES (whose FP32 dots see one row
    tile and several, full and ragged column groups): the solve converges to
    the solution found with the vectors in memory (clusters), to its tolerance."""
    s = scenes.sphere_scene(level)
    rng = np.random.default_rng(31)
    d = rng.standard_normal((12, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    W = np.exp(2j * np.pi * rng.random((R, 12)))
    out = []
    for mode in (solver, 3):
        c = api.Context.from_scene(s, n_pade=8, osrc_solver=mode, r_eps=0.1)
        c.set_transducer(3.0 * d, -d, np.full(12, 0.1), 2.6)
        c.set_excitations(W)
        rep = c.solve(precision=api.FP32, tol=1e-8, restart=100, operator_mode=1, batch_rhs=R, block_gmres=1)
        assert rep["converged"], rep
        out.append(np.stack([c.solution(r) for r in range(R)]))
        c.close()
    for r in range(R):
        assert rel(out[0][r], out[1][r]) < 1e-6, r


@pytest.mark.parametrize("precision,R", [("FP32", 1), ("FP64", 1), ("FP32", 3)])
@pytest.mark.parametrize("name", ["sphere", "two", "ribs"])
def test_products_back_to_back(api, name, precision, R):
    """A chain of products, each on the one before, without the host waiting
    in between: the same bits as with a wait after each (the kernels of a
    product start before the ones they follow have ended)."""
    import torch
    s = {"sphere": lambda: scenes.sphere_scene(3), "two": lambda: scenes.two_sphere_scene(1),
         "ribs": lambda: scenes.rib_scene(h=9e-3, freq=0.03e6)}[name]()
    x0 = torch.from_numpy(np.stack([scenes.smooth_trace_vector(s, r) for r in range(R)])).cuda()
    x0 = x0[0] if R == 1 else x0
    c = api.Context.from_scene(s)
    runs = []
    for wait in (True, False):
        x = x0
        for _ in range(8):
            y = c.apply(x, precision=getattr(api, precision))
            if wait:
                torch.cuda.synchronize()
            x = y / 2.0 ** 10
        torch.cuda.synchronize()
        runs.append(x.cpu().numpy())
    assert np.isfinite(runs[0]).all()
    assert np.array_equal(runs[0], runs[1])
    c.close()


@pytest.mark.parametrize("precision", ["FP32", "FP64", "BF16X3", "FP64_ASSEMBLED"])
def test_new_material_after_use(api, precision):
    """A domain's material changed after products of every kind: the next
    product is that of a context made with it (near field, far field and both
    assembled operators).  The assembled operators are summed by atomics."""
    p = getattr(api, precision)
    old, new = scenes.two_sphere_scene(1), scenes.two_sphere_scene(1, k2=4.4 + 0.3j, rho2=1.2)
    x = scenes.smooth_trace_vector(old, 3)
    c = api.Context.from_scene(new)
    ref = c.apply(x, precision=p)
    c.close()
    c = api.Context.from_scene(old)
    for q in (api.FP32, api.FP64, api.BF16X3, api.FP64_ASSEMBLED):
        before = c.apply(x, precision=q)
    assert rel(before, ref) > 1e-2
    c.set_material(1, new.domains[1].k, new.domains[1].rho)
    assert rel(c.apply(x, precision=p), ref) < (1e-12 if "64" in precision else 1e-6)
    c.close()


def test_loose_solves_of_two_sizes_at_once(api):
    """Contexts solving in four threads, whose largest domains (2,562 and 2,068
    vertices) take the same instance of the shared-memory preconditioner solver
    with different amounts of shared memory: no launch of either is refused,
    however the threads interleave."""
    import threading
    import torch
    sc = [scenes.sphere_scene(4)] + [scenes.kidney_scene(h=6e-3, freq=0.05e6)] * 3
    ctx = [api.Context.from_scene(s, stream=torch.cuda.Stream().cuda_stream) for s in sc]
    errors = []

    def work(c):
        try:
            for _ in range(20):
                c.solve(precision=api.FP32, tol=1e-14, operator_mode=1, max_iter=100)
        except Exception as e:  # a refused launch
            errors.append(e)

    for c in ctx:
        c.set_plane_wave((0, 0, 1))
        c.solve(precision=api.FP32, tol=1e-2, operator_mode=1, max_iter=20)  # set-up
    threads = [threading.Thread(target=work, args=(c,)) for c in ctx]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for c in ctx:
        c.close()
    assert not errors, errors


def test_fp64_assembled_digits_by_columns(api):
    """20,484 unknowns (a CTA's run covers a whole row tile): a smooth vector,
    and rows whose terms all add up over one half of the columns and cancel
    over the other, against 128-bit sums of the entries (products with unit
    vectors: one term, whose digits are exact).  A term loses 7 digit products
    of weight 2^-70 with digits of about 37 (rms), of either sign: 2^-58,
    against a largest term of 2^-4 within its 256 columns.  Six deviations of
    512 of them, and those of the units in quadrature; nothing from the sums."""
    import torch
    s = scenes.sphere_scene(5)
    c = api.Context.from_scene(s)
    N = c.n_dofs
    rows = np.array([0, 137, 2561, 5000, 10241, 10242, 15000, N - 1])
    idx = torch.from_numpy(rows).cuda()
    A = np.empty((len(rows), N), dtype=np.complex128)
    col = np.empty(N)  # largest part of each column
    for b in range(0, N, 1024):
        e = min(N, b + 1024)
        E = torch.zeros(e - b, N, dtype=torch.complex128, device="cuda")
        E[torch.arange(e - b), torch.arange(b, e)] = 1
        Y = c.apply(E, precision=api.FP64_ASSEMBLED)
        A[:, b:e] = Y[:, idx].T.cpu().numpy()
        col[b:e] = torch.view_as_real(Y).abs().amax(dim=(1, 2)).cpu().numpy()
    c0 = 2.0 ** np.ceil(np.log2(col))
    X = np.exp(-1j * np.angle(A))
    X[:, N // 2:] *= -1
    X = np.concatenate([X, scenes.smooth_trace_vector(s, 2)[None]])
    Y = c.apply(X, precision=api.FP64_ASSEMBLED)
    c.close()
    units = np.arange(0, N, 256)
    L = np.longdouble
    for r, i in enumerate(rows):
        for v in (r, len(rows)):
            ar, ai, xr, xi = (z.astype(L) for z in (A[r].real, A[r].imag, X[v].real, X[v].imag))
            dr = abs((ar * xr - ai * xi).sum() - L(Y[v, i].real))
            di = abs((ar * xi + ai * xr).sum() - L(Y[v, i].imag))
            largest = np.maximum.reduceat(np.abs(A[r]) / c0, units) * np.maximum.reduceat(np.abs(X[v]) * c0, units) * 4
            bound = 6 * np.sqrt(512) * 2.0 ** -54 * np.linalg.norm(largest)  # (4: powers of two above both)
            assert max(dr, di) < bound, (i, v, float(max(dr, di)), bound)


@pytest.mark.parametrize("name,R", [("ribs", 4), ("kidney", 6)])
def test_tensor_core_far_field_error(api, name, R):
    """The same product to the accuracy of its numbers: FP32 evaluation of the
    phase, 1/r and the gradient factor is good to a few 2^-23 of a term, the
    FP16 pairs keep 2^-21 of it, and the sums are rounded to nearest per
    source tile: together 2^-18 leaves a factor of four."""
    s = {"ribs": lambda: scenes.rib_scene(h=9e-3, freq=0.03e6), "kidney": lambda: scenes.kidney_scene(h=7.5e-3, freq=0.04e6)}[name]()
    c = api.Context.from_scene(s)
    X = np.stack([scenes.smooth_trace_vector(s, r) for r in range(R)])
    Y = c.apply(X, precision=api.FP32)
    Z = c.apply(X, precision=api.FP64)
    c.close()
    for r in range(R):
        assert rel(Y[r], Z[r]) < 2.0 ** -18, r


@pytest.mark.parametrize("level", [2, 3])
def test_fp64_assembled_hypersingular_rows(api, level):
    """W keeps FP64's rounding in the double-float assembly.  Without a
    wavenumber its rows add up to zero whatever the errors of V, because a
    source triangle's three curls do; what is left is the rounding of its terms
    and their sums, FP64 in the native assembly as well: at most twice that
    one's, on average over the rows (sums by atomics: the order differs)."""
    s = scenes.sphere_scene(level, k0=1e-9, k1=1e-9)
    left = []
    for native in (0, 1):
        c = api.Context.from_scene(s, fp64_far=native)
        N = c.n_dofs
        A = c.apply(np.eye(N, dtype=np.complex128), precision=api.FP64_ASSEMBLED).T
        c.close()
        W = A[N // 2:, N // 2:].real.astype(np.longdouble)
        left.append(np.mean(np.abs(W.sum(axis=1)) / np.sqrt((W ** 2).sum(axis=1))))
    assert left[0] < 2 * left[1], [float(v) for v in left]


@pytest.mark.parametrize("name,R", [("sphere", 1), ("sphere", 9), ("two", 2), ("two", 16), ("two1", 3), ("two1", 12)])
def test_fp64_assembled_digits_short_runs(api, name, R):
    """One block of 32 columns in all (24 unknowns), two (48), and runs of two
    and four blocks that start inside a unit of 256 columns and whose pieces
    make up a row tile (168): by the product's own columns, whose digits are
    exact, to 2^-54 of the largest scaled entry of a row and of a vector; rows
    here range over less than 2^12."""
    s = {"sphere": lambda: scenes.sphere_scene(0), "two": lambda: scenes.two_sphere_scene(0),
         "two1": lambda: scenes.two_sphere_scene(1)}[name]()
    c = api.Context.from_scene(s)
    A = c.apply(np.eye(c.n_dofs, dtype=np.complex128), precision=api.FP64_ASSEMBLED).T
    X = np.stack([scenes.smooth_trace_vector(s, r) for r in range(R)])
    Y = c.apply(X if R > 1 else X[0], precision=api.FP64_ASSEMBLED).reshape(R, -1)
    c.close()
    for r in range(R):
        assert rel(Y[r], A @ X[r]) < 1e-12
