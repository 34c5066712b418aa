"""The parallel-tempering decisions on energies of the size real systems have: large
common offsets, where a pair's difference is a few units in the last place of the
energies' leading binary32 part, and differences that put the exponent near 0 and near
the point below which no uniform accepts."""
import numpy as np
import pytest

import oracle
from paper_1204_6192_gb300 import hsg, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__
    __graft_entry__.build()


def ladder(kind, R_T):
    if kind == "wide":
        return inputs.geometric_temperatures(0.1, 1.0, R_T)
    return 1.0 + 1e-6 * np.arange(R_T)       # close: beta differences of 1e-6


def draw(rng, offset, spread, n):
    """Energies about the offset; a third of them one of three values, a third on both
    sides of 1e-6 (|a| + |b|) from the offset (where binary64 takes over)."""
    E = offset + rng.normal(0, spread, n)
    at = rng.integers(3, size=n)
    E[at == 0] = (offset + spread * np.array([0.0, 0.3, -1.0]))[rng.integers(3, size=(at == 0).sum())]
    edge = 2e-6 * abs(offset) * rng.choice([-1, 1], n) * rng.choice([0.0, 0.5, 0.999999, 1.0, 1.000001, 2.0], n)
    E[at == 1] = offset + edge[at == 1]
    return E


@pytest.mark.parametrize("ladder_kind", ["wide", "close"])
@pytest.mark.parametrize("offset,spread", [(-3e6, 0.1), (-3e6, 3.0), (-3e6, 100.0), (-3e6, 1e6), (-2.5e5, 1.0),
                                           (7e8, 20.0), (0.0, 1e-20)])
@pytest.mark.parametrize("R_T,R_O", [(5, 7), (32, 4), (97, 3)])
def test_pt_decisions_at_large_energies(R_T, R_O, offset, spread, ladder_kind):
    temps = ladder(ladder_kind, R_T)
    smp = inputs.Sample(L=4, J=np.zeros((64, 3)), H=None, temps=temps)
    ctx = hsg.Context([smp], R_O, 9)
    o = oracle.OracleSim([smp], R_O, 9).samples[0]
    rng = np.random.default_rng(R_T)
    accepted = 0
    for k in range(20):
        E = draw(rng, offset, spread, R_T * R_O)
        ctx.pt_exchange_energies(E)
        accepted = accepted + o.pt(E, k)
        np.testing.assert_array_equal(ctx.get_perm()[0], o.perm)
    np.testing.assert_array_equal(ctx.pt_stats()[0][0], accepted)
    moved, tunnel, _ = ctx.pt_diagnostics()
    np.testing.assert_array_equal(moved[0], o.moved)
    np.testing.assert_array_equal(tunnel[0], o.tunnel)
    ctx.close()
