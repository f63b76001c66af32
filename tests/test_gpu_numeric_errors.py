"""What is not a number ends in the stated status: a zero or non-finite LU pivot, and a forced flip whose ratio
is not finite, which is not taken.  No index in these kernels depends on a floating-point value.
"""
import numpy as np
import pytest

import oracle
from paper_2506_09611_gb300 import inputs
from tests.test_gpu_parity import FP64_TOL, make, rel

pytestmark = pytest.mark.gpu

afqmc = pytest.importorskip("paper_2506_09611_gb300.afqmc")

ERR_NUMERIC = -4


def _init_fails(L, ns, P, precision):
    X = inputs.initial_fields(2, L * L, seed=11)
    with afqmc.Context(2, precision=precision, stab_every=2, seed=11) as ctx:
        with pytest.raises(afqmc.AfqmcError) as e:
            ctx.init_walkers([L], [ns], [ns], np.concatenate([P.ravel(), P.ravel()]), X)
            ctx.measure_energy()
        assert e.value.code == ERR_NUMERIC


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("bad", [0.0, np.nan, np.inf])
@pytest.mark.parametrize("L,ns,col", [(4, 7, 0), (4, 7, 6), (9, 33, 31), (9, 33, 32), (33, 401, 200)])
def test_bad_pivot_is_reported(L, ns, col, bad, precision):
    """A zero or non-finite column of the trial state, in the first, a middle and the last column of a 32-column
    panel and beside a trailing update; the device then still serves a good walker."""
    P = inputs.trial_state(L, L, ns)
    P[:, col] = bad
    _init_fails(L, ns, P, precision)
    ctx, w, _, _ = make(4, 7, 2, stab=2)
    with ctx:
        for s in range(2):
            assert rel(ctx.G(0, s), w.G[s]) < FP64_TOL
        assert ctx.measure_energy()[1][0] == w.sign


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("value", [np.inf, np.nan])
@pytest.mark.parametrize("mode,k,nb", [("delayed", 16, 1), ("delayed", 5, 1), ("blockfb", 1, 4), ("blockfb", 1, 16)])
def test_forced_flip_without_a_ratio_is_not_taken(mode, k, nb, value, precision):
    """One diagonal element of G is not finite; its site alone is forced to flip."""
    L, ns, site = 4, 7, 9
    N = L * L
    ctx, _, _, _ = make(L, ns, 2, stab=2, precision=precision)
    with ctx:
        ctx.sweep_slice(1, +1, "delayed", k=16)
        G = ctx.G(0, 0)
        G[site, site] = value
        ctx.set_G(0, 0, G)
        before = ctx.fields(0)
        rep = np.zeros(2 * N, np.uint8)
        if mode == "blockfb":  # every proposal is the present field but the site's
            rep[:N] = before[0] > 0
            rep[site] ^= 1
            rep[N:] = 1
        else:
            rep[site] = 1
        ctx.sweep_slice(1, -1, mode, k=k, nb=nb, replay=rep)  # backward: decisions first, then the wrap
        np.testing.assert_array_equal(ctx.fields(0), before)
        dec = ctx.decisions(0)
        assert dec[N + site // nb if mode == "blockfb" else site] == 0
        with pytest.raises(afqmc.AfqmcError) as e:
            ctx.measure_energy()
        assert e.value.code == ERR_NUMERIC
