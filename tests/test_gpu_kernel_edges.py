"""Kernels at the sizes where they can go wrong: edges of tiles, remainders, the ends of the ranges that
choose between variants. Against the FP64 oracles, numpy's eigenvalues, or the library's general path.

Tolerances: FP64 results 1e-10 relative (max norm) as everywhere in these tests; the mixed mode's W
2e-3; eigenvalues 10 n eps |A| (backward stability of the Householder reduction and of the Sturm
counts); FNO outputs 1e-4 and gradients 2e-3 (FP32 sums of O(B N^3) terms)."""
import numpy as np
import pytest

from conftest import rel_err
from oracle import fno as ofno
from oracle import mixed, spectrum, tdh
from test_gpu_fno import _bf16, _pack, _unpack  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2205_06690_gb300 import binding
    binding.load()
    return binding


def _orbitals(N, box, count, seed):
    """A potential and `count` orthonormal smooth fields (no eigenstates: the kernels need none)."""
    rng = np.random.default_rng(seed)
    k = np.fft.fftfreq(N) * N
    soft = np.exp(-(k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :] ** 2) / 9.0)
    f = np.fft.ifftn(soft * np.fft.fftn(rng.standard_normal((count + 1, N, N, N)), axes=(1, 2, 3)), axes=(1, 2, 3)).real
    q, _ = np.linalg.qr(f[:count].reshape(count, -1).T)
    v = -2.0 * np.abs(f[count]) / np.max(np.abs(f[count]))
    return v, (q.T / (box / N) ** 1.5).reshape(count, N, N, N), np.sort(rng.standard_normal(count))


def _apply(B, precision, N, box, v, phi, eps, n_occ, n_o, n_c, prm, pairs, **options):
    with B.Context(0, precision) as c:
        for name, value in options.items():
            B.sbse_set_option(c.h, getattr(B, name), value)
        c.set_grid(N, box, v)
        c.set_orbitals(n_occ, n_o, n_c, phi, eps, 0.5)
        return c.apply_W(prm, pairs, copy_out=True)


def _check_w(B, N, n_occ, n_o, pairs, n_s, clean, steps=4):
    box = 0.4 * N
    v, phi, eps = _orbitals(N, box, n_occ + 1, N + n_occ)
    prm = B.TDHParams(n_s=n_s, n_steps=steps, clean_every=clean, dt=0.05, gamma=0.1, alpha=1e-4, seed=5)
    coeff = tdh.stochastic_coefficients(prm.seed, n_s, n_occ, "gaussian")
    op = tdh.TDHParams(n_steps=steps, dt=0.05, gamma=0.1, alpha=1e-4, clean_every=clean)
    ref = tdh.screened_potentials(tdh.Grid(N, box), v, phi, n_occ, n_o, coeff, op, pairs=pairs)
    ref = np.stack([ref[p].ravel() for p in pairs])
    assert rel_err(_apply(B, B.SBSE_FP64, N, box, v, phi, eps, n_occ, n_o, 1, prm, pairs), ref) < 1e-10
    assert rel_err(_apply(B, B.SBSE_MIXED, N, box, v, phi, eps, n_occ, n_o, 1, prm, pairs), ref) < 2e-3


@pytest.mark.parametrize("N", [18, 25, 27, 30, 36, 45, 50, 54, 60])
def test_further_grid_edges_match_oracle(B, N):
    """Odd pair count (the last Poisson slot packs one density), cleaning inside the run."""
    _check_w(B, N, 3, 2, [(0, 0), (0, 1), (1, 1)], 3, 2)


@pytest.mark.parametrize("n_occ,n_pairs,n_s", [(1, 1, 1), (4, 1, 3), (5, 3, 3), (64, 3, 5), (67, 6, 3)])
def test_fp64_cleaning_edges_match_oracle(B, n_occ, n_pairs, n_s):
    """Occupied counts and columns around the 4 x 4 overlap tiles, the 8 columns and 64 states of the
    update; 10^3 points leave the last chunk and the last tile of 128 points partly filled."""
    n_o = 1 if n_pairs == 1 else 3
    _check_w(B, 10, n_occ, n_o, tdh.pair_list(n_o)[:n_pairs], n_s, 1)


@pytest.mark.parametrize("N,n_o,count", [(16, 1, 1), (16, 4, 10), (32, 2, 3), (32, 5, 15), (40, 2, 3), (48, 1, 1),
                                         (48, 4, 9), (64, 2, 3)])
def test_bare_potentials_of_few_and_many_slots(B, N, n_o, count):
    """Both sides of the rule that gives a pencil four lanes (FP64, in the init; the slots of FP32 in
    one propagation step)."""
    box = 0.3 * N
    v, phi, eps = _orbitals(N, box, n_o + 1, N)
    pairs = tdh.pair_list(n_o)[:count]
    ref = np.stack([tdh.coulomb_periodic(phi[i] * phi[j], tdh.Grid(N, box)).ravel() for i, j in pairs])
    with B.Context(0, B.SBSE_FP64) as c:
        c.set_grid(N, box, v)
        c.set_orbitals(n_o, n_o, 1, phi, eps, 0.5)
        B.sbse_bare_W(c.h, pairs)
        assert rel_err(B.sbse_get_W(c.h, pairs, N ** 3), ref) < 1e-10
    prm = B.TDHParams(n_s=2, n_steps=1, clean_every=0, dt=0.05, gamma=0.1, alpha=1e-4, seed=1)
    coeff = tdh.stochastic_coefficients(1, 2, n_o, "gaussian")
    op = tdh.TDHParams(n_steps=1, dt=0.05, gamma=0.1, alpha=1e-4, clean_every=0)
    w = tdh.screened_potentials(tdh.Grid(N, box), v, phi, n_o, n_o, coeff, op, pairs=pairs[:1])
    for prec, tol in ((B.SBSE_FP64, 1e-10), (B.SBSE_MIXED, 2e-3)):
        assert rel_err(_apply(B, prec, N, box, v, phi, eps, n_o, n_o, 1, prm, pairs)[0], w[pairs[0]].ravel()) < tol


@pytest.mark.parametrize("N,n_pairs,n_s", [(18, 15, 2), (24, 3, 3), (32, 3, 3), (32, 21, 1), (40, 6, 1), (48, 3, 2),
                                           (48, 10, 1), (64, 1, 2), (64, 6, 1)])
def test_two_sweep_step_of_few_and_many_pairs(B, N, n_pairs, n_s):
    """Both sides of the rules that sum the density in the z sweep, with and without bulk copies."""
    n_o, box = 6, 0.4 * N
    pairs = tdh.pair_list(n_o)[:n_pairs]
    v, phi, eps = _orbitals(N, box, n_o + 1, N)
    prm = B.TDHParams(n_s=n_s, n_steps=2, clean_every=0, dt=0.05, gamma=0.1, alpha=1e-4, seed=3)
    coeff = tdh.stochastic_coefficients(prm.seed, n_s, n_o, "gaussian")
    op = tdh.TDHParams(n_steps=2, dt=0.05, gamma=0.1, alpha=1e-4, clean_every=0)
    ref = tdh.screened_potentials(tdh.Grid(N, box), v, phi, n_o, n_o, coeff, op, pairs=pairs)
    ref = np.stack([ref[p].ravel() for p in pairs])
    for tma in (0, 1):
        w = _apply(B, B.SBSE_MIXED, N, box, v, phi, eps, n_o, n_o, 1, prm, pairs, SBSE_OPT_TMA_PLANES=tma)
        assert rel_err(w, ref) < 2e-3


def _eig_noalloc(B, a, k):
    torch = pytest.importorskip("torch")
    d, ev = torch.from_numpy(np.ascontiguousarray(a)).cuda(), torch.empty(k, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    B.sbse_spectrum_noalloc(d.data_ptr(), a.shape[0], k, ev.data_ptr(), 0)
    return ev.cpu().numpy()


def _sym(n, kind):
    rng = np.random.default_rng(n)
    a = rng.standard_normal((n, n))
    a = 0.5 * (a + a.T)
    if kind == "diagonal":
        a = np.diag(np.diag(a))
    elif kind == "blocks":  # decoupled halves, one of them a multiple of the identity
        h = n // 2
        a[:h, h:] = a[h:, :h] = 0.0
        a[h:, h:] = 0.25 * np.eye(n - h)
    elif kind == "zero":
        a[:] = 0.0
    elif kind == "large":
        a *= 1e150
    elif kind == "small":
        a *= 1e-150
    return a


@pytest.mark.parametrize("n", [1, 2, 3, 4, 7, 15, 16, 17, 31, 33, 64, 100, 127, 128, 129, 255, 257, 512])
@pytest.mark.parametrize("kind", ["dense", "blocks"])
def test_eigenvalues_at_cluster_edges(B, n, kind):
    a = _sym(n, kind)
    k = min(n, 12)
    ref = np.linalg.eigvalsh(a)
    assert np.max(np.abs(_eig_noalloc(B, a, k) - ref[:k])) <= 10 * n * 2.2e-16 * max(1e-300, np.max(np.abs(ref)))


@pytest.mark.parametrize("kind", ["diagonal", "zero", "large", "small"])
def test_eigenvalues_of_special_matrices(B, kind):
    a = _sym(40, kind)
    ref = np.linalg.eigvalsh(a)
    assert np.max(np.abs(_eig_noalloc(B, a, 40) - ref)) <= 10 * 40 * 2.2e-16 * max(1e-11, np.max(np.abs(ref)))


@pytest.fixture(scope="module")
def wide(B):
    """An exchange-only A of 24 x 28 = 672 rows on 16^3: beyond the shared memory of the eigensolver's
    cluster, and more rows than four per SM for the spectrum."""
    N, box, n_o, n_c = 16, 8.0, 24, 28
    v, phi, eps = _orbitals(N, box, n_o + n_c, 2)
    c = B.Context(0, B.SBSE_FP64)
    c.set_grid(N, box, v)
    c.set_orbitals(n_o, n_o, n_c, phi, eps, 0.5)
    A = c.build_A(B.SBSE_EXCHANGE)
    yield c, A, phi, N, box, n_o, n_c
    c.close()


def test_eigenvalues_and_vectors_beyond_shared_memory(B, wide):
    c, A, n = wide[0], wide[1], wide[1].shape[0]
    ref = np.linalg.eigvalsh(0.5 * (A + A.T))
    tol = 10 * n * 2.2e-16 * np.max(np.abs(ref))
    assert np.max(np.abs(c.spectrum(6) - ref[:6])) <= tol
    ev, X = c.spectrum(6, vectors=True)
    assert np.max(np.abs(ev - ref[:6])) <= tol
    assert np.max(np.abs(A @ X - X * ev)) <= 1e-9 * np.max(np.abs(ref)) and np.max(np.abs(X.T @ X - np.eye(6))) <= 1e-9


def _chebyshev(A, f0, K, s, omega):
    c, w = spectrum.scaling(A)
    R = spectrum.residues(A, f0, K)
    return spectrum.sigma_chebyshev(R, c, w, omega, s), R


def test_absorption_of_wide_matrix(B, wide):
    c, A, phi, N, box, n_o, n_c = wide
    f0 = spectrum.dipoles(tdh.Grid(N, box), phi[:n_o], phi[n_o:], 1)
    omega = np.linspace(0.1, 4.0, 37)
    ref, R = _chebyshev(A, f0, 65, 0.1, omega)
    sig, res = c.absorption(1, 65, 0.1, omega)
    assert rel_err(res, R) < 1e-8 and rel_err(sig, ref) < 1e-8
    ref, R = _chebyshev(A, f0, 2050, 0.1, omega)  # enough terms for rounds of four
    sig, res = c.absorption(1, 2050, 0.1, omega)
    assert rel_err(res, R) < 1e-8 and rel_err(sig, ref) < 1e-8


@pytest.mark.parametrize("n_o,n_c,terms", [(1, 1, 2), (1, 3, 3), (3, 11, 64), (5, 13, 257), (1, 3, 63),
                                          (1, 7, 64), (4, 8, 66), (5, 13, 65), (13, 10, 127)])
def test_absorption_of_small_matrices(B, n_o, n_c, terms):
    """One block, a row count that is no multiple of a warp's or block's rows, few terms."""
    N, box = 10, 6.0
    v, phi, eps = _orbitals(N, box, n_o + n_c, n_o)
    omega = np.linspace(0.1, 4.0, 5)
    with B.Context(0, B.SBSE_FP64) as c:
        c.set_grid(N, box, v)
        c.set_orbitals(n_o, n_o, n_c, phi, eps, 0.5)
        A = c.build_A(B.SBSE_EXCHANGE)
        if n_o * n_c == 1:  # Gershgorin discs of one row leave no interval to scale
            return
        sig, res = c.absorption(0, terms, 0.2, omega)
    f0 = spectrum.dipoles(tdh.Grid(N, box), phi[:n_o], phi[n_o:], 0)
    ref, R = _chebyshev(A, f0, terms, 0.2, omega)
    assert rel_err(res, R) < 1e-8 and rel_err(sig, ref) < 1e-8


@pytest.mark.parametrize("n_occ,n_o,n_c", [(1, 1, 1), (7, 4, 9), (9, 5, 8), (33, 3, 2)])
def test_hole_grid_projections(B, n_occ, n_o, n_c):
    """Window and basis counts around the 4 x 8 tiles; a basis of fewer rows takes more chunks."""
    N, box = 10, 5.0
    v, phi, eps = _orbitals(N, box, n_occ + n_c, n_occ)
    g = tdh.Grid(N, box)
    po = phi[n_occ - n_o:n_occ]
    W = {(i, j): tdh.coulomb_periodic(po[i] * po[j], g) for i, j in tdh.pair_list(n_o)}
    f = np.random.default_rng(1).standard_normal((n_o, N, N, N))
    with B.Context(0, B.SBSE_FP64) as c:
        c.set_grid(N, box, v)
        c.set_orbitals(n_occ, n_o, n_c, phi, eps, 0.5)
        B.sbse_bare_W(c.h, tdh.pair_list(n_o))
        for proj, cond in ((B.SBSE_Q_OCCUPIED, False), (B.SBSE_Q_CONDUCTION, True)):
            op = mixed.MixedA(g, v, phi, eps, n_occ, n_o, n_c, W, 0.5, conduction_only=cond)
            fq = op.Q(f)
            got = B.sbse_apply_A_mixed(c.h, proj, fq.reshape(n_o, -1)).reshape(fq.shape)
            assert rel_err(got, op(fq)) < 1e-10


@pytest.mark.parametrize("N,C,m,L,batch", [(9, 5, 4, 2, 2), (10, 33, 5, 2, 1), (13, 3, 6, 1, 9), (8, 64, 2, 2, 11),
                                           (70, 2, 3, 1, 1)])
def test_fno_edges_match_oracle(B, N, C, m, L, batch):
    """Odd grids, every mode kept, channel counts off the compiled ones, batches beyond the mix's
    registers and shared memory, planes of more rows than one tile."""
    torch = pytest.importorskip("torch")
    net = B.FNO(N, width=C, modes=m, layers=L, max_batch=batch)
    vec = _pack(ofno.init_params(C, m, L, seed=N))
    net.set_params(vec)
    pr = _unpack(vec, C, m, L, round_bf16=True)
    rng = np.random.default_rng(1)
    x = rng.standard_normal((batch, 2, N, N, N)).astype(np.float32)
    dy = rng.standard_normal((batch, N, N, N)).astype(np.float32)
    xd, dyd = torch.from_numpy(x).cuda(), torch.from_numpy(dy).cuda()
    yd = torch.empty((batch, N, N, N), dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    net.forward(batch, xd.data_ptr(), yd.data_ptr())
    y, cache = ofno.forward(pr, x.astype(np.float64), m, keep=True)
    assert rel_err(yd.cpu().numpy(), y) < 1e-4
    net.gradients(batch, xd.data_ptr(), dyd.data_ptr())
    gp, ref = _unpack(net.get_params()[1], C, m, L), ofno.backward(pr, cache, dy.astype(np.float64), m)
    for name in ("lift_w", "lift_b", "proj_w"):
        assert rel_err(getattr(gp, name), ref[name]) < 2e-3
    assert abs(gp.proj_b - ref["proj_b"]) < 2e-3 * max(1.0, abs(ref["proj_b"]))
    for name in ("pw_w", "pw_b", "spec"):
        for a, b in zip(getattr(gp, name), ref[name]):
            assert rel_err(a, b) < 2e-3
    net.close()


def test_fno_planes_beyond_shared_memory(B):
    """Planes whose folded transforms do not fit take the direct sums: forward only, one channel."""
    torch = pytest.importorskip("torch")
    N, C, m, L = 168, 1, 84, 1
    net = B.FNO(N, width=C, modes=m, layers=L, max_batch=1)
    vec = _pack(ofno.init_params(C, m, L, seed=1))
    net.set_params(vec)
    x = np.random.default_rng(1).standard_normal((1, 2, N, N, N)).astype(np.float32)
    xd, yd = torch.from_numpy(x).cuda(), torch.empty((1, N, N, N), dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    net.forward(1, xd.data_ptr(), yd.data_ptr())
    assert rel_err(yd.cpu().numpy(), ofno.forward(_unpack(vec, C, m, L, round_bf16=True), x.astype(np.float64), m)) < 1e-4
    net.close()


def test_absorption_without_interval_is_not_finite(B):
    """One row leaves no interval to scale: the vectors are NaN, and the call says so instead of waiting."""
    N, box = 10, 6.0
    v, phi, eps = _orbitals(N, box, 2, 1)
    with B.Context(0, B.SBSE_FP64) as c:
        c.set_grid(N, box, v)
        c.set_orbitals(1, 1, 1, phi, eps, 0.5)
        c.build_A(B.SBSE_EXCHANGE)
        for terms, omega in ((2, 1.0), (70, 1.0), (70, 1e3)):  # (far from every Gaussian as well)
            with pytest.raises(B.SbseError) as e:
                c.absorption(0, terms, 0.2, np.array([omega]))
            assert e.value.code == B.SBSE_ERR_NUMERIC


def test_absorption_at_a_memory_limit(B):
    """A context without room for the matrix squares (10 MiB at 462 rows) takes single terms: it needs no
    more than the vectors above what few terms need, and gives the same spectrum."""
    N, box, n_o, n_c, few, many = 10, 6.0, 21, 22, 63, 1024
    v, phi, eps = _orbitals(N, box, n_o + n_c, 3)
    omega = np.linspace(0.1, 4.0, 5)
    n = n_o * n_c

    def least(terms):
        with B.Context(0, B.SBSE_FP64) as c:
            c.set_grid(N, box, v)
            c.set_orbitals(n_o, n_o, n_c, phi, eps, 0.5)
            c.build_A(B.SBSE_EXCHANGE)
            for limit in range(1, 200):
                B.sbse_set_option(c.h, B.SBSE_OPT_MEM_LIMIT_MB, limit)
                try:
                    at_limit = c.absorption(0, terms, 0.2, omega)
                except B.SbseError as e:
                    assert e.code == B.SBSE_ERR_OOM
                    continue
                break
        with B.Context(0, B.SBSE_FP64) as c:
            c.set_grid(N, box, v)
            c.set_orbitals(n_o, n_o, n_c, phi, eps, 0.5)
            c.build_A(B.SBSE_EXCHANGE)
            free = c.absorption(0, terms, 0.2, omega)
        assert all(rel_err(a, b) < 1e-8 for a, b in zip(at_limit, free))
        return limit

    assert least(many) <= least(few) + ((n + 6) * (many - few) * 8 >> 20) + 2


@pytest.mark.parametrize("N,C,batch", [(9, 5, 2), (24, 33, 1), (32, 64, 1)])
def test_fno_bias_gradient_of_cancelling_fields(B, N, C, batch):
    """Sums that cancel to a small part of their terms: rounded to FP32 once (2^-23), after pairs of floats
    over at most 1024 points (1024 2^-46 of the absolute sum)."""
    torch = pytest.importorskip("torch")
    net = B.FNO(N, width=C, modes=2, layers=1, max_batch=batch)
    net.set_params(_pack(ofno.init_params(C, 2, 1, seed=N)))
    rng = np.random.default_rng(N)
    dy = rng.standard_normal((batch, N, N, N))
    dy = (dy - dy.mean() + 1e-4 / N ** 3).astype(np.float32)
    xd, dyd = torch.zeros((batch, 2, N, N, N), device="cuda"), torch.from_numpy(dy).cuda()
    torch.cuda.synchronize()
    net.gradients(batch, xd.data_ptr(), dyd.data_ptr())
    got, ref = float(net.get_params()[1][-1]), float(dy.sum(dtype=np.float64))
    assert abs(got - ref) <= 2.0 ** -23 * abs(ref) + 2.0 ** -36 * float(np.abs(dy).sum(dtype=np.float64))
    net.close()


@pytest.mark.parametrize("N,C,batch", [(9, 5, 2), (16, 32, 1), (24, 33, 3)])
def test_fno_bias_gradients_add_in_order(B, N, C, batch):
    """Bias gradients are the FP32 sums of 4096 points in a row, chunks joined in FP64, to the bit (one chunk
    that is not full, a full one, a full one and a remainder across batch entries; 5, 32 and 33 rows), and keep
    an infinite entry."""
    torch = pytest.importorskip("torch")
    net = B.FNO(N, width=C, modes=2, layers=1, max_batch=batch)
    vec = _pack(ofno.init_params(C, 2, 1, seed=N))
    net.set_params(vec)
    w = vec[-1 - C:-1]  # the projection: dL/dU of the only layer is w[c] dy
    xd = torch.zeros((batch, 2, N, N, N), device="cuda")

    def bias(dy):
        d = torch.from_numpy(dy).cuda()
        torch.cuda.synchronize()
        net.gradients(batch, xd.data_ptr(), d.data_ptr())
        g = net.get_params()[1]
        return np.append(g[-1 - 2 * C:-1 - C], g[-1])

    def in_order(x):
        return np.float32(sum(float(np.add.accumulate(x[k:k + 4096], dtype=np.float32)[-1]) for k in range(0, x.size, 4096)))

    dy = np.random.default_rng(N).standard_normal((batch, N, N, N)).astype(np.float32)
    ref = np.array([in_order((c * dy).ravel()) for c in np.append(w, np.float32(1))])
    exact = float(dy.sum(dtype=np.float64))
    assert abs(float(ref[-1]) - exact) < 2.0 ** -12 * abs(exact)  # (sums that keep their leading bits)
    assert np.array_equal(bias(dy), ref)
    dy[-1, 1, 2, 3] = np.inf
    assert np.array_equal(bias(dy), np.copysign(np.float32(np.inf), np.append(w, np.float32(1))))
    net.close()


@pytest.mark.parametrize("n", [1, 2, 3, 40, 257])
@pytest.mark.parametrize("where", ["all", "corner", "last", "inf"])
def test_eigenvalues_of_matrices_that_are_not_finite(B, n, where):
    """No eigenvalue comes out as a number, the zero of a vanishing matrix least of all."""
    a = _sym(n, "dense")
    if where == "all":
        a[:] = np.nan
    elif where == "corner":  # the first row and column stay finite
        a[n // 2:, n // 2:] = np.nan
    elif where == "last":
        a[n - 1, n - 1] = np.nan
    else:
        a[0, n - 1] = a[n - 1, 0] = np.inf
    assert np.all(np.isnan(_eig_noalloc(B, a, min(n, 12))))


def test_spectrum_of_a_diverged_surrogate_is_refused(B):
    """W fields that are NaN reach A unchecked; eigenvalues and vectors of it are a numeric error."""
    torch = pytest.importorskip("torch")
    N, box, n_o, n_c = 10, 6.0, 3, 4
    v, phi, eps = _orbitals(N, box, n_o + n_c, 4)
    pairs = tdh.pair_list(n_o)
    y = torch.full((len(pairs), N, N, N), float("nan"), device="cuda")
    torch.cuda.synchronize()
    with B.Context(0, B.SBSE_FP64) as c:
        c.set_grid(N, box, v)
        c.set_orbitals(n_o, n_o, n_c, phi, eps, 0.5)
        B.sbse_bare_W(c.h, pairs)
        B.sbse_add_W(c.h, pairs, y.data_ptr(), 1.0)
        c.build_A()
        for vectors in (False, True):
            with pytest.raises(B.SbseError) as e:
                c.spectrum(5, vectors=vectors)
            assert e.value.code == B.SBSE_ERR_NUMERIC


def test_fno_batch_beyond_a_grid_dimension(B):
    """More batch entries than blocks in gridDim.y (65535): outputs and gradients are those of the same entries
    in two parts (gradients: FP32 sums of 65605 terms in another grouping, sqrt(65605) 2^-24 = 1.5e-5 and a margin)."""
    torch = pytest.importorskip("torch")
    N, C, m, L, batch, part = 4, 2, 2, 2, 65535 + 70, 40000
    gen = torch.Generator(device="cuda").manual_seed(1)
    xd = torch.randn((batch, 2, N, N, N), generator=gen, device="cuda")
    dyd = 1.0 + torch.randn((batch, N, N, N), generator=gen, device="cuda")
    vec = _pack(ofno.init_params(C, m, L, seed=2))

    def run(first, count):
        net = B.FNO(N, width=C, modes=m, layers=L, max_batch=count)
        net.set_params(vec)
        x, dy, y = xd[first:first + count], dyd[first:first + count], torch.empty((count, N, N, N), device="cuda")
        torch.cuda.synchronize()
        net.forward(count, x.data_ptr(), y.data_ptr())
        net.gradients(count, x.data_ptr(), dy.data_ptr())
        g = net.get_params()[1].astype(np.float64)
        net.close()
        return y, g

    y, g = run(0, batch)
    (y0, g0), (y1, g1) = run(0, part), run(part, batch - part)
    assert torch.equal(y, torch.cat([y0, y1]))
    assert rel_err(g, g0 + g1) < 1e-4


def test_hole_grid_operator_at_a_memory_limit(B):
    """At 4 rows the operator holds at most 18 FP64 fields (2 MiB each on 64^3) besides the context's own: six for
    the operator, two vectors and two packed slots of two. Counted from the four fields of the boundary
    potential."""
    N, box, n_o, n_c = 64, 16.0, 4, 1
    v, phi, eps = _orbitals(N, box, n_o + n_c, 5)
    pairs = tdh.pair_list(n_o)
    w = np.random.default_rng(2).standard_normal((len(pairs), N ** 3))
    f = np.random.default_rng(3).standard_normal((n_o, N ** 3))

    def least(call):
        with B.Context(0, B.SBSE_FP64) as c:
            c.set_grid(N, box, v)
            c.set_orbitals(n_o, n_o, n_c, phi, eps, 0.5)
            B.sbse_set_W(c.h, pairs, w)
            for limit in range(1, 400):
                B.sbse_set_option(c.h, B.SBSE_OPT_MEM_LIMIT_MB, limit)
                try:
                    return limit, call(c.h)
                except B.SbseError as e:
                    assert e.code == B.SBSE_ERR_OOM

    first, _ = least(B.sbse_boundary_potential)
    operator, at_limit = least(lambda h: B.sbse_apply_A_mixed(h, B.SBSE_Q_OCCUPIED, f))
    assert operator - first <= 2 * (18 - 4) + 1
    with B.Context(0, B.SBSE_FP64) as c:
        c.set_grid(N, box, v)
        c.set_orbitals(n_o, n_o, n_c, phi, eps, 0.5)
        B.sbse_set_W(c.h, pairs, w)
        assert np.array_equal(at_limit, B.sbse_apply_A_mixed(c.h, B.SBSE_Q_OCCUPIED, f))


@pytest.mark.parametrize("N,n_occ,n_o", [(16, 5, 1), (16, 6, 4), (32, 5, 3), (40, 5, 4), (48, 3, 2),  # four lanes per pencil
                                         (9, 4, 2), (15, 4, 3), (54, 3, 1),                   # runtime radix
                                         (18, 4, 3), (20, 6, 4), (45, 3, 2), (32, 8, 8)])     # a thread per pencil
def test_hole_grid_operator_of_every_round_trip(B, N, n_occ, n_o):
    """Kinetic multiplier of the rows' slots and Coulomb kernel of the last slot in each of the z passes, with
    odd and even row counts."""
    box = 0.4 * N
    v, phi, eps = _orbitals(N, box, n_occ + 1, N + n_o)
    g = tdh.Grid(N, box)
    po = phi[n_occ - n_o:n_occ]
    pairs = tdh.pair_list(n_o)
    W = {(i, j): tdh.coulomb_periodic(po[i] * po[j], g) for i, j in pairs}
    op = mixed.MixedA(g, v, phi, eps, n_occ, n_o, 1, W, 0.5, conduction_only=False)
    f = op.Q(np.random.default_rng(N).standard_normal((n_o, N, N, N)))
    with B.Context(0, B.SBSE_FP64) as c:
        c.set_grid(N, box, v)
        c.set_orbitals(n_occ, n_o, 1, phi, eps, 0.5)
        B.sbse_bare_W(c.h, pairs)
        got = B.sbse_apply_A_mixed(c.h, B.SBSE_Q_OCCUPIED, f.reshape(n_o, -1)).reshape(f.shape)
    assert rel_err(got, op(f)) < 1e-10


@pytest.mark.parametrize("scale", [1e-150, 1e-100, 1e100])
@pytest.mark.parametrize("n", [2, 3, 40, 257])
def test_eigenvalues_of_scaled_matrices(B, n, scale):
    """Relative to the matrix's own norm, however small: a solver that returns zeros does not pass."""
    a = scale * _sym(n, "dense")
    ref = np.linalg.eigvalsh(a)
    assert np.max(np.abs(_eig_noalloc(B, a, min(n, 12)) - ref[:12])) <= 10 * n * 2.2e-16 * np.max(np.abs(ref))


def test_eigenvalues_of_the_zero_matrix(B):
    assert np.array_equal(_eig_noalloc(B, np.zeros((40, 40)), 12), np.zeros(12))


@pytest.mark.parametrize("N,n_pairs", [(32, 18), (32, 19), (48, 8), (48, 9), (64, 4), (64, 5), (80, 3), (80, 4), (96, 3)])
def test_streamed_z_sweep_gives_the_bits_of_plain_loads(B, N, n_pairs):
    """The z sweep fed by bulk copies (from 608 blocks of a pair's 32 columns on) and the one with plain loads
    sum the same density terms in the same order; below the rule both options take the plain sweep."""
    n_o, box = 6, 0.4 * N
    pairs = tdh.pair_list(n_o)[:n_pairs]
    v, phi, eps = _orbitals(N, box, n_o + 1, N)
    prm = B.TDHParams(n_s=3, n_steps=5, clean_every=3, dt=0.05, gamma=0.1, alpha=1e-4, seed=3)
    w = [_apply(B, B.SBSE_MIXED, N, box, v, phi, eps, n_o, n_o, 1, prm, pairs, SBSE_OPT_TMA_PLANES=tma) for tma in (0, 1)]
    assert np.array_equal(w[0], w[1])


def test_fno_holds_no_fields_of_the_direct_sums(B):
    """A network whose transforms are folded allocates nothing for the direct sums (34 MB here): parameters and
    their copies, activations, spectra and one field of the z transform."""
    torch = pytest.importorskip("torch")
    N, C, m, L, batch = 64, 32, 8, 1, 4
    warm = B.FNO(8, width=2, modes=2, layers=1, max_batch=1)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    net = B.FNO(N, width=C, modes=m, layers=L, max_batch=batch)
    used = free - torch.cuda.mem_get_info()[0]
    act, modes, direct = batch * C * N ** 3 * 4, 4 * m ** 3, batch * C * N * N * m * 8
    need = (L + 1 + L + 3) * act + (L + 1) * batch * C * modes * 8 + batch * C * N * 2 * m * m * 8 + 18 * net.n_params + \
        2 * batch * N ** 3 * 4
    assert used < need + direct // 2
    net.close()
    warm.close()


def test_absorption_residues_keep_64_bits(B):
    """Residues of many terms against the recursion in extended precision, on the library's own A: within one
    rounding (2^-53) per term, root mean square."""
    N, box, n_o, n_c, terms = 12, 6.0, 10, 11, 2048
    v, phi, eps = _orbitals(N, box, n_o + n_c, 7)
    with B.Context(0, B.SBSE_FP64) as c:
        c.set_grid(N, box, v)
        c.set_orbitals(n_o, n_o, n_c, phi, eps, 0.5)
        A = c.build_A(B.SBSE_EXCHANGE)
        _, res = c.absorption(0, terms, 0.2, np.linspace(0.1, 4.0, 5))
    f0 = spectrum.dipoles(tdh.Grid(N, box), phi[:n_o], phi[n_o:], 0).astype(np.longdouble)
    mid, half = spectrum.scaling(A)
    m = (A.astype(np.longdouble) - np.longdouble(mid) * np.eye(len(A))) / np.longdouble(half)
    prev, cur = f0, m @ f0
    ref = [f0 @ prev, f0 @ cur]
    for _ in range(2, terms):
        prev, cur = cur, 2 * (m @ cur) - prev
        ref.append(f0 @ cur)
    ref = np.array(ref)
    assert np.sqrt(np.sum((res - ref) ** 2) / np.sum(ref ** 2)) <= terms * 2.0 ** -53
