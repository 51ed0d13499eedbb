"""The packed engines beside the other calls of a chain, and where they end: a chain
in a batch and then alone."""
import numpy as np
import pytest

from paper_1303_6016_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_1303_6016_gb300 import build, gfmc
    build.build()
    gfmc.load()
    return gfmc


@pytest.mark.parametrize("L,team,wide", [(8, 12, 16), (18, 96, 108), (20, 130, 140)])
def test_chain_alone_after_a_team_smaller_than_its_engine(G, L, team, wide):
    """FP64 chains whose packed engine takes more CTAs (wide) than their tiles (8, 91,
    125) and than a team they ran on before: after the team, the chain alone gives
    bit for bit what it gives after a team of as many CTAs as its engine."""
    n = 4
    sp = inputs.uniform_sphere(L, 2)
    kw = dict(M=16, beta=12.0, mu=-2.0, seed=5)
    with G.Chain(L, sp, **kw) as a, G.Chain(L, sp, **kw) as b:
        ba, bb = G.run_batch([a], n, team_ctas=[team]), G.run_batch([b], n, team_ctas=[wide])
        assert np.array_equal(ba[0]["decisions"], bb[0]["decisions"])
        ra, rb = a.updates(n), b.updates(n)
        assert np.array_equal(ra["d_omega"], rb["d_omega"])
        assert np.array_equal(ra["decisions"], rb["decisions"])
