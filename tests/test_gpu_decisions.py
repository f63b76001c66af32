"""FP32 decisions on their own: the ratios, proposals and accepts of the FP32 update kernels against the FP64
oracle, on replayed chains (every ratio that the kernel reports) and running free (every decision whose uniform
lies further from its threshold than the tolerance; the seeds leave no nearer one).

Tolerances.  FP32 G is within 1e-5 ||G||_F of the oracle's (FP32_TOL), ||G||_F < 10 at these sizes and
|Delta| = |e^{2 gamma} - 1| < 1.5, so a site's ratio s r_up r_dn, |r_up| + |r_dn| < 6, is within 1e-3 max(1, |R|),
and so is a proposal probability; a block's ratio is a product of at most n_b of them.
"""
import numpy as np
import pytest

import oracle
from paper_2506_09611_gb300 import inputs
from tests.test_gpu_parity import _replay, make

pytestmark = pytest.mark.gpu

afqmc = pytest.importorskip("paper_2506_09611_gb300.afqmc")

SITE_TOL = 1e-3


def _close(got, ref, tol):
    err = np.abs(got - ref) / np.maximum(1.0, np.abs(ref))
    assert np.all(err < tol), (np.argmax(err), err.max())


def _hs(U):
    return oracle.HS_SZ_REAL if U > 0 else oracle.HS_CHARGE_REAL


CASES = [(9, 36, "local", 1, 1, 4.0), (9, 36, "local", 1, 1, -4.0), (13, 80, "local", 1, 1, 4.0),
         (9, 36, "delayed", 33, 1, 4.0), (9, 36, "delayed", 128, 1, -4.0),
         (9, 36, "blockfb", 1, 1, 1.0), (9, 36, "blockfb", 1, 7, 4.0), (9, 36, "blockfb", 1, 16, 4.0),
         (9, 36, "blockfb", 1, 32, 4.0), (9, 36, "blockfb", 1, 16, -4.0), (9, 36, "blockfb", 1, 17, -4.0)]


@pytest.mark.parametrize("L,ns,mode,k,nb,U", CASES)
def test_reported_ratios_fp32(L, ns, mode, k, nb, U):
    """Two replayed slices."""
    N = L * L
    ctx, w, P, X = make(L, ns, 2, U=U, stab=2, precision="fp32", seed=17, hs=_hs(U))
    with ctx:
        for ell in (1, 2):
            dec, ratio, extra = w.sweep_slice(ell, +1, mode, inputs.uniforms(17, 0, ell - 1, 2 * N), k=k, nb=nb)
            if mode == "blockfb":
                rep = _replay(N, nb, dec, extra)
            else:
                rep = np.concatenate([dec, np.zeros(N)]).astype(np.uint8)
            ctx.sweep_slice(ell, +1, mode, k=k, nb=nb, replay=rep)
            got = ctx.ratios(0)
            if mode == "blockfb":
                _close(got[:N], extra["lam_plus"], SITE_TOL)
                _close(got[N:N + len(dec)], ratio, nb * SITE_TOL)
            else:
                _close(got[:N], ratio, SITE_TOL)


@pytest.mark.parametrize("L,ns,mode,k,nb,U", CASES)
def test_free_decisions_fp32(L, ns, mode, k, nb, U):
    """One slice with the device's own uniforms."""
    N = L * L
    for seed in range(1, 40):
        ctx, w, P, X = make(L, ns, 2, U=U, stab=2, precision="fp32", seed=seed, hs=_hs(U))
        with ctx:
            u = inputs.uniforms(seed, 0, 0, 2 * N)
            dec, ratio, extra = w.sweep_slice(1, +1, mode, u, k=k, nb=nb)
            if mode == "blockfb":
                near = np.abs(u[:N] - extra["lam_plus"]) < SITE_TOL
                near_block = np.abs(u[N:N + len(dec)] - np.abs(ratio)) < nb * SITE_TOL * np.maximum(1.0, np.abs(ratio))
                near_block &= ratio != 1.0  # no flip proposed: always accepted
            else:
                near, near_block = np.abs(u[:N] - np.abs(ratio)) < SITE_TOL * np.maximum(1.0, np.abs(ratio)), False
            if np.any(near) or np.any(near_block):
                continue
            ctx.sweep_slice(1, +1, mode, k=k, nb=nb)
            got = ctx.decisions(0)
            if mode == "blockfb":
                np.testing.assert_array_equal(got[:N], extra["xprop"] > 0)
                np.testing.assert_array_equal(got[N:N + len(dec)], dec)
            else:
                np.testing.assert_array_equal(got[:N], dec)
            np.testing.assert_array_equal(ctx.fields(0), w.x)
            return
    pytest.fail("no seed leaves every uniform clear of its threshold")
