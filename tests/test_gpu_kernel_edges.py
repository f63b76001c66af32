"""Sizes at which the sweep's kernels change path: the register tiles of the window kernels (32, 64 and
128 sites) and of the stateless update, the register-resident local update and its fall-back, the
32-column panels of the FP64 LU and its solve, and the vectors per block of the lattice DFT.  FP64 runs
free against the FP64 oracle (equal decisions, G within 1e-10), FP32 replays the oracle's decisions (G
within 1e-5), as in the other parity tests.
"""
import numpy as np
import pytest

import oracle
from paper_2506_09611_gb300 import inputs
from tests import test_gpu_soc as gsoc
from tests.test_gpu_parity import FP32_TOL, FP64_TOL, _replay, _run_sweep, make, rel

pytestmark = pytest.mark.gpu

afqmc = pytest.importorskip("paper_2506_09611_gb300.afqmc")
soc = pytest.importorskip("paper_2506_09611_gb300.soc")


def _replay_sweep(L, ns, mode, k=1, nb=1, U=4.0, slices=2, keep=1.0):
    """Forward slices of an FP32 walker with the oracle's decisions forced; keep < 1 also turns that share
    of the accepts into rejections."""
    N = L * L
    ctx, w, P, X = make(L, ns, slices, U=U, stab=slices, precision="fp32", seed=17)
    rng = np.random.default_rng(3)
    with ctx:
        for ell in range(1, slices + 1):
            u = inputs.uniforms(17, 0, ell - 1, 2 * N)
            if keep < 1.0:
                rep = np.zeros(2 * N, np.uint8)
                rep[:N] = rng.random(N) < keep
                w.sweep_slice(ell, +1, mode, u, k=k, nb=nb, replay=rep[:N])
            else:
                dec, _, extra = w.sweep_slice(ell, +1, mode, u, k=k, nb=nb)
                if mode == "blockfb":
                    rep = _replay(N, nb, dec, extra)
                else:
                    rep = np.zeros(2 * N, np.uint8)
                    rep[:N] = dec
            ctx.sweep_slice(ell, +1, mode, k=k, nb=nb, replay=rep)
            for s in range(2):
                r = rel(ctx.G(0, s), w.G[s])
                assert r < FP32_TOL, (ell, s, r)
        np.testing.assert_array_equal(ctx.fields(0), w.x)


@pytest.mark.parametrize("k", [1, 31, 32, 33, 63, 64])
def test_delayed_windows_fp64(k):
    """N = 81: every k leaves a ragged last window, and odd starts of the later ones."""
    ctx, w, P, X = make(9, 36, 2, stab=2)
    with ctx:
        _run_sweep(ctx, w, "delayed", k=k, stab=2)


@pytest.mark.parametrize("L,k", [(9, 1), (9, 31), (9, 33), (13, 64), (13, 65), (13, 127), (13, 128)])
def test_delayed_windows_fp32(L, k):
    _replay_sweep(L, (L * L) // 2 - 3, "delayed", k=k)


@pytest.mark.parametrize("nb", [1, 2, 15, 16, 17, 31, 32])
def test_block_force_bias_fp32(nb):
    """Blocks of the 16- and 32-lane kernels; 81 sites leave a ragged window and a ragged block."""
    _replay_sweep(9, 36, "blockfb", nb=nb, U=1.0)


@pytest.mark.parametrize("nb", [17, 32])
def test_block_force_bias_fp64(nb):
    ctx, w, P, X = make(9, 36, 2, U=1.0, stab=2)
    with ctx:
        _run_sweep(ctx, w, "blockfb", nb=nb, stab=2)


@pytest.mark.parametrize("L,ns", [(2, 1), (13, 80), (29, 401), (30, 431), (32, 489), (41, 800)])
def test_local_update_fp32(L, ns):
    """One or more rows per CTA, 3, 6 and 11 rows per thread, and (41 x 41) G kept in global memory."""
    _replay_sweep(L, ns, "local", slices=1)


@pytest.mark.parametrize("L,ns", [(13, 80), (30, 431)])
def test_local_update_sparse_accepts_fp32(L, ns):
    """Accepts further apart than the rows published ahead."""
    _replay_sweep(L, ns, "local", slices=1, keep=0.15)


@pytest.mark.parametrize("L,ns", [(9, 1), (9, 31), (9, 32), (9, 33), (9, 64), (9, 65), (17, 100), (27, 203), (33, 401)])
def test_factorisation_and_solve(L, ns):
    """G(0) and a recompute: LU panels and solves with whole and partial 32-blocks, one to several CTAs per
    matrix, and (33 x 33) trailing updates beside the next panel until they are too small."""
    ctx, w, P, X = make(L, ns, 2, stab=1)
    with ctx:
        for s in range(2):
            assert rel(ctx.G(0, s), w.G[s]) < FP64_TOL
        ctx.sweep_slice(1, +1, "delayed", k=16)
        w.sweep_slice(1, +1, "delayed", inputs.uniforms(11, 0, 0, 2 * L * L), k=16)
        ctx.recompute_G()
        w.recompute(1)
        for s in range(2):
            assert rel(ctx.G(0, s), w.G[s]) < FP64_TOL
        assert ctx.measure_energy()[1][0] == w.sign  # pivots and the parity of the row permutations


@pytest.mark.parametrize("pad", [0, 1, 4])
@pytest.mark.parametrize("precision,m", [("fp64", 1), ("fp64", 32), ("fp64", 33), ("fp64", 64), ("fp32", 1),
                                         ("fp32", 31), ("fp32", 64), ("fp32", 65), ("fp32", 128)])
def test_apply_flips_register_tiles(precision, m, pad):
    """Against the dense formula in FP64.  The error of a partially pivoted m x m elimination is bounded by
    m eps cond(M) (growth aside); 64 eps cond(M) covers it and the products at these sizes."""
    torch = pytest.importorskip("torch")
    N = 150
    rng = np.random.default_rng(m)
    dt = torch.float64 if precision == "fp64" else torch.float32
    Q = np.linalg.qr(rng.standard_normal((N, N // 2)))[0]
    G = torch.zeros(2, N, N + pad, dtype=dt, device="cuda")
    G[:, :, :N] = torch.from_numpy(np.eye(N) - Q @ Q.T).to(dt)
    sites = rng.permutation(N)[:m].astype(np.int32)
    delta = np.exp(rng.choice([-1.0, 1.0], 2 * m)) - 1.0
    ref, tol = [], []
    for s in range(2):
        G0 = G[s, :, :N].double().cpu().numpy()
        D = np.diag(delta[s * m:(s + 1) * m])
        M = np.eye(m) + (np.eye(m) - G0[np.ix_(sites, sites)]) @ D
        ref.append(G0 - G0[:, sites] @ D @ np.linalg.solve(M, np.eye(N)[sites] - G0[sites]))
        tol.append(64 * (2.3e-16 if precision == "fp64" else 1.2e-7) * np.linalg.cond(M))
    sites_d, delta_d = torch.from_numpy(sites).cuda(), torch.from_numpy(delta).cuda()
    afqmc.afqmc_apply_flips(precision, N, N + pad, G[0].data_ptr(), G[1].data_ptr(), sites_d.data_ptr(),
                            delta_d.data_ptr(), m, torch.cuda.current_stream())
    for s in range(2):
        assert rel(G[s, :, :N].double().cpu().numpy(), ref[s]) < tol[s]


@pytest.mark.parametrize("spin", [0, 1])
def test_apply_flips_singular_spin_changes_nothing(spin):
    """1 + (1 - G_ii) Delta = 0 in one spin only: reported, and neither G is touched."""
    torch = pytest.importorskip("torch")
    N = 8
    G = torch.eye(N, dtype=torch.float64, device="cuda").repeat(2, 1, 1) * 0.5
    before = G.clone()
    delta = torch.tensor([1.0, 1.0], dtype=torch.float64)
    delta[spin] = -2.0
    sites, dev = torch.tensor([3], dtype=torch.int32, device="cuda"), delta.cuda()
    with pytest.raises(afqmc.AfqmcError):
        afqmc.afqmc_apply_flips("fp64", N, N, G[0].data_ptr(), G[1].data_ptr(), sites.data_ptr(), dev.data_ptr(), 1,
                                torch.cuda.current_stream())
    assert torch.equal(G, before)


@pytest.mark.parametrize("L,ns", [(2, 1), (3, 4), (5, 11), (20, 60)])
def test_pairing_dft_sizes(L, ns):
    """The momentum-space matrices against numpy's FFT of the same G (Mk: its definition on a sample of
    momenta)."""
    N = L * L
    ctx = soc.SocContext(L, 1, 2 * ns, 1, "fp64", "tc3", 1, 1.0, 0.0, -4.0, 0.05, 7, hs="sz")
    with ctx:
        ctx.init(inputs.sz_trial_state(L, ns), inputs.initial_fields(1, N, seed=7))
        got = ctx.measure_pairing()
        G = ctx.G(0)
    # <c+_j c_i> = delta_ij - G_ij at (i, j); F2 A F2^+ with F_qj = e^{-i q r_j} / L
    A = (np.eye(2 * N) - G).reshape(2, L, L, 2, L, L)
    At = np.fft.ifft2(np.fft.fft2(A, axes=(1, 2)), axes=(4, 5)).reshape(2 * N, 2 * N)
    np.testing.assert_allclose(got["nk"][0], np.diag(At), atol=1e-11)
    rng = np.random.default_rng(L)
    for k, kp in rng.integers(0, N, (200, 2)):
        mk, mkp = [(-(q // L) % L) * L + (-(q % L)) % L for q in (k, kp)]
        ref = At[kp, k] * At[N + mkp, N + mk] - At[N + mkp, k] * At[kp, N + mk]
        assert abs(got["Mk"][0][k, kp] - ref) < 1e-11


@pytest.mark.parametrize("mode,k,nb", [("blockfb", 1, 15), ("blockfb", 1, 16), ("blockfb", 1, 17), ("blockfb", 1, 32),
                                       ("delayed", 16, 1), ("delayed", 32, 1)])
def test_soc_window_inverse(mode, k, nb):
    """Window matrices up to and beyond the 32 x 32 register tile, with a ragged last window (36 sites)."""
    ctx, w = gsoc.make(6, 36, 2, 1, seed=23)
    with ctx:
        gsoc._free_run(ctx, w, mode, k, nb, 23, 4, 1, FP64_TOL)
