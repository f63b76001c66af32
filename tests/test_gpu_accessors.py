"""get_G returns what set_G put in, element by element, on both sides of the size up to which it is packed on the
host (100 KB of the padded G) and with odd leading dimensions."""
import numpy as np
import pytest

from paper_2506_09611_gb300 import inputs

pytestmark = pytest.mark.gpu

afqmc = pytest.importorskip("paper_2506_09611_gb300.afqmc")
soc = pytest.importorskip("paper_2506_09611_gb300.soc")


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("L", [2, 5, 10, 11, 12, 13])
def test_G_round_trip(L, precision):
    N, n, rng = L * L, 2, np.random.default_rng(L)
    ns = N // 2
    P = inputs.trial_state(L, L, ns)
    X = np.concatenate([inputs.initial_fields(2, N, seed=1, walker=j).ravel() for j in range(n)])
    with afqmc.Context(2, precision=precision, stab_every=2, seed=1) as ctx:
        ctx.init_walkers([L] * n, [ns] * n, [ns] * n, np.concatenate([P.ravel(), P.ravel()] * n), X)
        G = rng.standard_normal((n, 2, N, N)).astype(np.float64 if precision == "fp64" else np.float32)
        for j in range(n):
            for s in range(2):
                ctx.set_G(j, s, G[j, s])
        for j in range(n):
            for s in range(2):
                np.testing.assert_array_equal(ctx.G(j, s), G[j, s])


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("L", [2, 5, 6, 7, 8])
def test_soc_G_round_trip(L, precision):
    N, n, rng = L * L, 2, np.random.default_rng(L)
    X = np.concatenate([inputs.initial_fields(2, N, seed=1 + j).ravel() for j in range(n)])
    ctx = soc.SocContext(L, 2, 2 * (N // 2), n, precision, "tc3", 2, 1.0, 0.0, -4.0, 0.05, 1, hs="sz")
    with ctx:
        ctx.init(inputs.sz_trial_state(L, N // 2), X)
        dt = np.complex128 if precision == "fp64" else np.complex64
        G = (rng.standard_normal((n, 2 * N, 2 * N)) + 1j * rng.standard_normal((n, 2 * N, 2 * N))).astype(dt)
        for j in range(n):
            ctx.set_G(j, G[j])
        for j in range(n):
            np.testing.assert_array_equal(ctx.G(j), G[j])
