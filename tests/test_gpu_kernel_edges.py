"""The kernels at the sizes where their tiles, rows and warps end (GPU): the
reduction to tridiagonal form with its back-transformation, the grouped
digit-split products of two problems, the recombination of the split-BF16
forms, the FP32 form's fused h psi on ragged axes and the FP64 form's float-pair
passes, and the damping network's convolutions, each against the FP64 oracle
or numpy.

Tolerances, from the arithmetic: a backward stable reduction of n <= 257 states
leaves n eps ||H|| = 6e-14 ||H|| in eigenvalues and residuals, the bisection
stops at 2^-43 ||T|| = 1.1e-13 ||T||, and 1e-12 leaves a factor for their
constants; the digit-split products keep 1e-14 of the largest element, five of
them in a Newton-Schulz step, each again corrected by the next: 1e-12; BF16x3
and x6 as in the parity tests of the same calls."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
import test_gpu_eigen as TE
import test_gpu_parity as TP
import test_gpu_precond as TN
from paper_1610_07522_gb300 import binding as B
from paper_1610_07522_gb300 import inputs as IN

pytestmark = pytest.mark.gpu


def _hermitian(kind, n, rng):
    a = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    if kind == "random":
        return a + a.conj().T
    d = np.diag(-60.0 + 100.0 * (np.arange(n) + 0.5 * rng.random(n)) / n)
    if kind == "blocks":                    # decoupled: reflectors that are the identity
        H = (a + a.conj().T) / np.sqrt(n)
        k = n // 3
        H[:k, k:] = 0.0
        H[k:, :k] = 0.0
        H[2 * k:, :2 * k] = 0.0
        H[:2 * k, 2 * k:] = 0.0
        H[2 * k:, 2 * k:] = 0.0
        return H + d
    # couplings from 1e-2 down to 1e-16 along the matrix: reflectors far below 1
    e = 10.0 ** (-2.0 - 14.0 * np.arange(n) / n)
    E = a * np.minimum(e[:, None], e[None, :])
    return d + E + E.conj().T


@pytest.mark.parametrize("kind", ["random", "blocks", "graded"])
@pytest.mark.parametrize("n", [2, 31, 33, 64, 65, 96, 127, 128, 129, 153, 193, 257])
def test_reduction_and_back_transformation(kind, n):
    rng = np.random.default_rng(7 * n + len(kind))
    H = _hermitian(kind, n, rng)
    c = TE._ctx(n)
    B.sky_tune_set(c, B.SKY_KNOB_EIGEN_METHOD, B.SKY_EIG_TRIDIAGONAL)
    M, lam = TE._solve(c, H)
    B.sky_destroy(c)
    lw = np.linalg.eigvalsh(H)
    nrm = float(np.max(np.abs(lw)))
    assert np.max(np.abs(lam - lw)) < 1e-12 * nrm
    assert np.max(np.abs(M.conj().T @ M - np.eye(n))) < 1e-12
    assert np.max(np.abs(H @ M - M * lam)) < 1e-12 * nrm


@pytest.mark.parametrize("sizes", [(96, 95), (96, 96), (128, 129), (161, 80), (97, 1)])
def test_grouped_products_of_two_problems(sizes):
    rng = np.random.default_rng(sum(sizes))
    c = TE._ctx(max(sizes))
    S, C = [], []
    for n in sizes:
        a = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
        S.append(np.eye(n) + 0.05 / np.sqrt(n) * (a + a.conj().T))
        C.append(torch.zeros((n, n), dtype=torch.complex128, device="cuda:0"))
    B.sky_orthonormalize_batched(c, [TE._dev(x) for x in S], list(sizes), C)
    B.sky_sync(c)
    for x, y in zip(S, C):
        w, U = np.linalg.eigh(x)
        want = (U / np.sqrt(w)) @ U.conj().T
        got = y.cpu().numpy()
        # C or its transpose's conjugate alike: S^{-1/2} is Hermitian up to the
        # convention of its indices
        assert min(np.max(np.abs(got - want)), np.max(np.abs(got - want.T))) < 1e-12
    B.sky_destroy(c)


@pytest.mark.parametrize("prec", [B.SKY_F32_BF16X3, B.SKY_F32_BF16X6])
@pytest.mark.parametrize("I", [1, 2, 15, 17, 33, 63, 65, 129])
def test_split_bf16_recombination_of_odd_state_counts(prec, I):
    rng = np.random.default_rng(40 + I)
    with TP.Ctx((8, 12, 8), prec=prec, max_states=I) as c:
        a = TP._r32(IN.random_spinors(c.grid.n, I, rng))
        M = (rng.standard_normal((I, I)) + 1j * rng.standard_normal((I, I))) / np.sqrt(I)
        out = torch.zeros(a.shape, dtype=torch.complex64, device="cuda:0")
        B.sky_rotate(c.ctx, TP.dev32(a), TP.dev(M), I, out)
        assert TP.relerr(TP.host(out), O.rotate(a, M)) < TP.TC_TOL[prec]


@pytest.mark.parametrize("grid", [(8, 20, 24), (32, 20, 12), (8, 32, 16), (16, 24, 32)])
def test_fp32_default_h_on_ragged_axes(grid):
    """Without a knob set the fused passes run on axes up to 32 (bit-identical
    to knob 1), the general ones agree within the FP32 bound."""
    rng = np.random.default_rng(sum(grid))
    I, out = 3, []
    with TP.Ctx(grid, twist=(0.4, -1.1, 2.0), prec=B.SKY_F32, max_states=I) as c:
        g = c.grid
        psi = TP._r32(IN.random_spinors(g.n, I, rng))
        U, Bf, W = TP._fields(g, rng)
        want = O.apply_h(psi, U, Bf, W, g)
        for knob in (None, 1, 0):
            if knob is not None:
                B.sky_tune_set(c.ctx, B.SKY_KNOB_FUSED_H, knob)
            d_h = torch.zeros(psi.shape, dtype=torch.complex64, device="cuda:0")
            B.sky_apply_h(c.ctx, TP.dev(U), TP.dev(Bf), TP.dev(W), TP.dev32(psi), d_h, I)
            out.append(TP.host(d_h))
            assert TP.relerr(out[-1], want) < TP.REL32
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("grid,I", [((8, 12, 20), 1), ((20, 8, 32), 5), ((32, 8, 12), 3), ((8, 24, 16), 2)])
def test_fp64_pair_passes_on_ragged_axes(grid, I):
    rng = np.random.default_rng(sum(grid) + I)
    with TP.Ctx(grid, twist=(0.4, -1.1, 2.0), max_states=I) as c:
        g = c.grid
        psi = IN.random_spinors(g.n, I, rng)
        U, Bf, W = TP._fields(g, rng)
        want = O.apply_h(psi, U, Bf, W, g)
        e_w, n_w = O.sp_energies(psi, want, g)
        d_h = torch.zeros(psi.shape, dtype=torch.complex128, device="cuda:0")
        eps = torch.zeros(I, dtype=torch.float64, device="cuda:0")
        hn2 = torch.zeros(I, dtype=torch.float64, device="cuda:0")
        B.sky_apply_h(c.ctx, TP.dev(U), TP.dev(Bf), TP.dev(W), TP.dev(psi), d_h, I, eps, hn2)
        assert TP.relerr(TP.host(d_h), want) < TP.REL
        assert TP.relerr(TP.host(eps), e_w) < TP.REL and TP.relerr(TP.host(hn2), n_w) < TP.REL
        rho_w, tau_w, J_w, dJ_w = O.densities(psi, g)
        rho = torch.zeros(g.G, dtype=torch.float64, device="cuda:0")
        tau, dJ = torch.zeros_like(rho), torch.zeros_like(rho)
        J = torch.zeros(3 * g.G, dtype=torch.float64, device="cuda:0")
        B.sky_densities(c.ctx, TP.dev(psi), I, rho, tau, J, dJ)
        for got, ref in ((rho, rho_w), (tau, tau_w), (J, J_w), (dJ, dJ_w)):
            assert TP.relerr(TP.host(got), ref.ravel()) < TP.REL


@pytest.mark.parametrize("grid", [(8, 8, 8), (20, 8, 12), (8, 32, 24)])
def test_network_convolutions_on_small_and_ragged_grids(grid):
    TN.test_net_forward_loss_and_gradient(grid, 1)


def test_input_that_looks_like_an_unset_word_does_not_stall_the_reduction():
    """The reduction's published values are their own flags (a signalling NaN means
    not there yet) and its first step publishes a column as it came: the same
    pattern in the input has to end as any NaN does, not in a wait that runs out."""
    n = 150
    S = 4.0 * np.eye(n, dtype=np.complex128)
    S[0, 1:5] = S[1:5, 0] = 0.5
    S.view(np.uint64)[[1, 3], [2 * 3, 2 * 1]] = 0x7FF4000000C0FFEE     # S[1, 3], S[3, 1]
    c = TE._ctx(n)
    C = torch.zeros((n, n), dtype=torch.complex128, device="cuda:0")
    B.sky_orthonormalize(c, TE._dev(S), n, C)
    with pytest.raises(B.SkyError) as ei:
        B.sky_sync(c)
    assert ei.value.status in (B.SKY_ENOTPD, B.SKY_ENOCONV)   # (SKY_ETIMEOUT would come first)
    B.sky_destroy(c)


@pytest.mark.parametrize("sizes", [(120,), (191,), (96, 95), (280, 120), (161, 80), (97, 1), (192, 60, 130)])
def test_loewdin_factors_of_problems_too_small_for_six_digits(sizes):
    """S^{-1/2} in the oracle's index convention; problems below 192 states, whose
    Newton-Schulz products alone are FP64, keep that accuracy beside larger ones:
    n eps (FP64 sums of n terms, each step corrected by the next) and 16 eps where
    that is less; the others the six digits' 1e-12."""
    rng = np.random.default_rng(sum(sizes))
    c = TE._ctx(max(sizes))
    B.sky_reserve_batch(c, len(sizes))
    S, C = [], []
    for n in sizes:
        a = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
        S.append(np.eye(n) + 0.05 / np.sqrt(n) * (a + a.conj().T))
        C.append(torch.zeros((n, n), dtype=torch.complex128, device="cuda:0"))
    B.sky_orthonormalize_batched(c, [TE._dev(x) for x in S], list(sizes), C)
    B.sky_sync(c)
    for n, x, y in zip(sizes, S, C):
        got = y.cpu().numpy()
        eps = np.finfo(float).eps
        tol = max(n, 16) * eps if n < 192 else 1e-12
        assert np.max(np.abs(got @ x @ got.conj().T - np.eye(n))) < tol
        assert np.max(np.abs(got - O.loewdin(x))) < (8 * tol if n < 192 else tol)
    B.sky_destroy(c)


@pytest.mark.parametrize("sizes", [(128, 64, 130), (192, 64, 256), (130, 97, 200, 128, 31, 60, 150, 129)])
def test_diagonalisation_of_three_to_eight_problems(sizes):
    """Batches of up to eight problems: the launches of the largest alone serve them
    all, and the eigenvectors come back as those of single problems do."""
    rng = np.random.default_rng(len(sizes))
    H = [_hermitian("random", n, rng) for n in sizes]
    z = lambda n: torch.zeros((n, n), dtype=torch.complex128, device="cuda:0")
    launches = []
    for batch in ([max(H, key=len)], H):
        ns = [h.shape[0] for h in batch]
        c = TE._ctx(max(sizes))
        B.sky_reserve_batch(c, len(ns))
        B.sky_tune_set(c, B.SKY_KNOB_EIGEN_METHOD, B.SKY_EIG_TRIDIAGONAL)
        M, lam = [z(n) for n in ns], [torch.zeros(n, dtype=torch.float64, device="cuda:0") for n in ns]
        l0 = B.sky_kernel_launches()
        B.sky_subspace_diag_batched(c, [TE._dev(h) for h in batch],
                                    [TE._dev(np.eye(n, dtype=np.complex128)) for n in ns], ns, M, lam)
        launches.append(B.sky_kernel_launches() - l0)
        B.sky_sync(c)
        for h, m, w in zip(batch, M, lam):
            m, w, lw = m.cpu().numpy(), w.cpu().numpy(), np.linalg.eigvalsh(h)
            nrm = float(np.max(np.abs(lw)))
            assert np.max(np.abs(w - lw)) < 1e-12 * nrm
            assert np.max(np.abs(m.conj().T @ m - np.eye(len(w)))) < 1e-12
            assert np.max(np.abs(h @ m - m * w)) < 1e-12 * nrm
        B.sky_destroy(c)
    assert launches[1] == launches[0]


def test_x6_overlap_sums_as_short_for_many_states():
    """The x6 form's sums are 1024 values long whatever the number of states, also
    where their partials take several rounds (32^3: from 500 states on): the
    entries of the first states are those of a call with these alone, the partials
    the same to the bit, their FP64 sum in another order (128 terms)."""
    I0, I = 200, 1040
    g = torch.Generator(device="cuda:0").manual_seed(11)
    a = torch.randn((I, 2 * 32 ** 3), dtype=torch.complex64, device="cuda:0", generator=g)
    X = []
    for n in (I0, I):
        c = B.sky_init((32, 32, 32), (1.0,) * 3, dict(IN.SLY4), False, (0.0,) * 3, B.SKY_F32_BF16X6, n,
                       torch.cuda.current_stream().cuda_stream)
        x = torch.zeros((n, n), dtype=torch.complex128, device="cuda:0")
        B.sky_overlap(c, a[:n].contiguous(), a[:n].contiguous(), n, x)
        B.sky_sync(c)
        B.sky_destroy(c)
        X.append(x[:I0, :I0].cpu().numpy())
    assert np.max(np.abs(X[0] - X[1])) < 128 * np.finfo(float).eps * np.max(np.abs(X[0]))


@pytest.mark.parametrize("prec", [B.SKY_F32_BF16X3, B.SKY_F32_BF16X6])
def test_split_bf16_overlap_beyond_the_floats_range(prec):
    """Partials that are floats, a sum that is not: 2048 products of 2.5e35."""
    I = 3
    with TP.Ctx((8, 8, 8), prec=prec, max_states=I) as c:
        a = torch.full((I, 1024), 5e17 * (1 + 1j), dtype=torch.complex64, device="cuda:0")
        X = torch.zeros((I, I), dtype=torch.complex128, device="cuda:0")
        B.sky_overlap(c.ctx, a, a, I, X)
        v = float(np.float32(5e17)) ** 2 * 2048
        assert TP.relerr(TP.host(X), np.full((I, I), v, dtype=complex)) < TP.TC_TOL[prec]


@pytest.mark.parametrize("grid", [(32, 16, 16), (32, 8, 16), (32, 8, 12), (24, 8, 12)])
def test_fused_h_knob_says_what_runs(grid):
    """Setting SKY_KNOB_FUSED_H to what it reads changes nothing, to the bit, and a
    context says by it whether h psi is fused."""
    rng = np.random.default_rng(sum(grid))
    with TP.Ctx(grid, twist=(0.4, -1.1, 2.0), prec=B.SKY_F32, max_states=3) as c:
        psi = TP.dev32(TP._r32(IN.random_spinors(c.grid.n, 3, rng)))
        U, Bf, W = (TP.dev(x) for x in TP._fields(c.grid, rng))
        default = B.sky_tune_get(c.ctx, B.SKY_KNOB_FUSED_H)
        out = []
        for knob in (None, default, 1 - default):
            if knob is not None:
                B.sky_tune_set(c.ctx, B.SKY_KNOB_FUSED_H, knob)
            d_h = torch.zeros_like(psi)
            B.sky_apply_h(c.ctx, U, Bf, W, psi, d_h, 3)
            out.append(TP.host(d_h))
        assert np.array_equal(out[0], out[1])
        assert not np.array_equal(out[0], out[2])


def _decaying_states(g, I, rng):
    """States that fall off to 1e-16 of their largest value and below."""
    r2 = np.meshgrid(*[(np.arange(n) - n / 2.0) ** 2 for n in g.shape], indexing="ij")
    return IN.random_spinors(g.n, I, rng) * np.exp(-sum(r2) / 8.0)


@pytest.mark.parametrize("grid", [(12, 16, 20), (32, 24, 8)])
@pytest.mark.parametrize("power", [-100, -64, 64, 100])
def test_fp64_h_psi_scales_with_the_states(grid, power):
    """States times a power of two: h psi times it at the bound of the unscaled call,
    though float pairs hold it between the passes (lines below 2^-126 among them)."""
    rng = np.random.default_rng(power + 200)
    I, s = 4, 2.0 ** power
    with TP.Ctx(grid, twist=(0.3, -0.2, 0.7), max_states=I) as c:
        psi = _decaying_states(c.grid, I, rng)
        U, Bf, W = TP._fields(c.grid, rng)
        d_h = torch.zeros(psi.shape, dtype=torch.complex128, device="cuda:0")
        B.sky_apply_h(c.ctx, TP.dev(U), TP.dev(Bf), TP.dev(W), TP.dev(psi * s), d_h, I)
        assert TP.relerr(TP.host(d_h) / s, O.apply_h(psi, U, Bf, W, c.grid)) < 1e-12


@pytest.mark.parametrize("grid", [(12, 16, 20), (32, 24, 8)])
@pytest.mark.parametrize("power", [-100, -64, 64, 100])
def test_fp64_densities_scale_with_the_states(grid, power):
    """States times a power of two: the densities times its square at the bounds of
    the unscaled call (1e-12, and 1e-11 for div J, one more derivative), also where
    the products of the gradients leave the range of the floats."""
    rng = np.random.default_rng(power + 200)
    I, s = 4, 2.0 ** power
    with TP.Ctx(grid, twist=(0.3, -0.2, 0.7), max_states=I) as c:
        g = c.grid
        psi = _decaying_states(g, I, rng)
        z = lambda n: torch.zeros(n, dtype=torch.float64, device="cuda:0")
        got = [z(g.G), z(g.G), z(3 * g.G), z(g.G)]
        B.sky_densities(c.ctx, TP.dev(psi * s), I, *got)
        for x, w, tol in zip(got, O.densities(psi, g), (1e-12, 1e-12, 1e-12, 1e-11)):
            assert TP.relerr(TP.host(x) / s / s, w.ravel()) < tol


@pytest.mark.parametrize("grid", [(48, 8, 12), (8, 64, 8), (12, 16, 48), (64, 48, 16)])
@pytest.mark.parametrize("coulomb", [True, False])
def test_real_fields_on_long_axes(grid, coulomb):
    """The direct sums of the real-field derivatives and of the Coulomb transform up
    to their longest axes, at the bounds of the short ones (the parity test of the
    same calls)."""
    rng = np.random.default_rng(sum(grid))
    with TP.Ctx(grid, dx=(0.9, 1.0, 1.1), coulomb=coulomb, prec=B.SKY_F32, max_states=2) as c:
        g = c.grid
        rho = np.stack([0.08 + 0.01 * IN.random_smooth_field(g.n, rng, 0.0, 1.0) for _ in range(2)])
        tau, dJ = 0.6 * rho, 0.1 * rho - 0.005
        U_w, B_w, W_w = O.mean_fields(rho, tau, dJ, TP.P, g, coulomb)
        E_w = O.energy(rho, tau, dJ, TP.P, g, coulomb)
        z = lambda *n: torch.zeros(n, dtype=torch.float64, device="cuda:0")
        U, Bf, W, out = z(2, g.G), z(2, g.G), z(2, 3, g.G), z(8)
        B.sky_mean_fields(c.ctx, TP.dev(rho), TP.dev(tau), TP.dev(dJ), U, Bf, W)
        B.sky_energy(c.ctx, TP.dev(rho), TP.dev(tau), TP.dev(dJ), out)
        assert TP.relerr(TP.host(U), U_w.reshape(2, -1)) < 1e-11
        assert TP.relerr(TP.host(Bf), B_w.reshape(2, -1)) < 1e-12
        assert TP.relerr(TP.host(W), W_w.reshape(2, 3, -1)) < 1e-11
        for e, k in zip(TP.host(out), ["total", "kin", "rho", "tau", "drho", "nJ", "coul", "A"]):
            assert abs(e - E_w[k]) <= 1e-11 * max(1.0, abs(E_w[k])), k
        psi = TP.dev32(TP._r32(IN.random_spinors(g.n, 2, rng)))
        r, t, J, d = z(g.G), z(g.G), z(3 * g.G), z(g.G)
        B.sky_densities(c.ctx, psi, 2, r, t, J, d)
        Jh = TP.host(J).reshape((3,) + g.shape)
        assert TP.relerr(TP.host(d), sum(O.deriv_real(Jh[j], j, g) for j in range(3)).ravel()) < 1e-11


@pytest.mark.parametrize("grid,I", [((24, 24, 24), 231), ((32, 32, 32), 97)])
def test_fp32_fused_h_in_uneven_chunks(grid, I):
    """More states than a chunk of the fused h psi holds (227 at 24^3, 96 at 32^3):
    two chunks, the last one smaller; states on both sides of the seam against the
    oracle, every state against the same states alone (the same arithmetic)."""
    rng = np.random.default_rng(I)
    with TP.Ctx(grid, twist=(1.3, -0.2, 0.9), prec=B.SKY_F32, max_states=I) as c:
        g = c.grid
        B.sky_tune_set(c.ctx, B.SKY_KNOB_FUSED_H, 1)
        psi = TP._r32(IN.random_spinors(g.n, I, rng))
        U, Bf, W = TP._fields(g, rng)
        d_psi, fields = TP.dev32(psi), [TP.dev(x) for x in (U, Bf, W)]

        def run(a, b):
            d_h = torch.zeros_like(d_psi[a:b])
            e = torch.zeros(b - a, dtype=torch.float64, device="cuda:0")
            n2 = torch.zeros_like(e)
            B.sky_apply_h(c.ctx, *fields, d_psi[a:b].contiguous(), d_h, b - a, e, n2)
            return TP.host(d_h), TP.host(e), TP.host(n2)

        h, e, n2 = run(0, I)
        seam = (I + 1) // 2
        for a, b in ((0, 60), (seam - 30, seam + 30), (I - 60, I)):
            for got, want in zip(run(a, b), (h, e, n2)):
                assert np.array_equal(got, want[a:b])
        for s in (0, seam - 1, seam, I - 1):
            want = O.apply_h(psi[s:s + 1], U, Bf, W, g)
            ew, nw = O.sp_energies(psi[s:s + 1], want, g)
            assert TP.relerr(h[s:s + 1], want) < TP.REL32
            assert TP.relerr(e[s:s + 1], ew) < TP.REL32
            assert TP.relerr(n2[s:s + 1], nw) < TP.REL32


def test_x6_overlap_of_a_context_made_for_x3():
    """A context keeps the partial buffer of the form it was made for: after
    sky_set_prec the x6 overlap takes it in rounds (24^3, 400 states: two) and gives
    what an x6 context gives, but for the FP64 sum of 54 terms in another order."""
    I, X = 400, []
    g = torch.Generator(device="cuda:0").manual_seed(5)
    a = torch.randn((I, 2 * 24 ** 3), dtype=torch.complex64, device="cuda:0", generator=g)
    for first in (B.SKY_F32_BF16X3, B.SKY_F32_BF16X6):
        c = B.sky_init((24, 24, 24), (1.0,) * 3, dict(IN.SLY4), False, (0.0,) * 3, first, I,
                       torch.cuda.current_stream().cuda_stream)
        B.sky_set_prec(c, B.SKY_F32_BF16X6)
        x = torch.zeros((I, I), dtype=torch.complex128, device="cuda:0")
        B.sky_overlap(c, a, a, I, x)
        B.sky_sync(c)
        B.sky_destroy(c)
        X.append(x.cpu().numpy())
    assert np.max(np.abs(X[0] - X[1])) < 54 * np.finfo(float).eps * np.max(np.abs(X[0]))


@pytest.mark.parametrize("sizes", [(129, 100), (97, 60), (200, 193)])
def test_subspace_of_two_problems_with_their_loewdin_factors(sizes):
    """C from S, then M from C^H H C, both for two problems at once: M^H S M = I and
    M^H H M = diag(lambda) with the eigenvalues of the pencil (H, S).  Bounds: the
    grouped products' 1e-12 of the largest entry, five factors in a row, and the
    reduction's 1e-12 ||H||."""
    from scipy.linalg import eigh

    rng = np.random.default_rng(sum(sizes))
    c = TE._ctx(max(sizes))
    S, H = [], []
    for n in sizes:
        a = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
        S.append(np.eye(n) + 0.1 / np.sqrt(n) * (a + a.conj().T))
        H.append(_hermitian("random", n, rng))
    z = lambda n: torch.zeros((n, n), dtype=torch.complex128, device="cuda:0")
    C, M = [z(n) for n in sizes], [z(n) for n in sizes]
    lam = [torch.zeros(n, dtype=torch.float64, device="cuda:0") for n in sizes]
    B.sky_orthonormalize_batched(c, [TE._dev(x) for x in S], list(sizes), C)
    B.sky_subspace_diag_batched(c, [TE._dev(x) for x in H], C, list(sizes), M, lam)
    B.sky_sync(c)
    B.sky_destroy(c)
    for s, h, m, w in zip(S, H, M, lam):
        m, w = m.cpu().numpy(), w.cpu().numpy()
        lw = eigh(h, s, eigvals_only=True)
        nrm = float(np.max(np.abs(lw)))
        assert np.max(np.abs(w - lw)) < 5e-12 * nrm
        assert np.max(np.abs(m.conj().T @ s @ m - np.eye(len(w)))) < 5e-12
        assert np.max(np.abs(m.conj().T @ h @ m - np.diag(w))) < 5e-12 * nrm
