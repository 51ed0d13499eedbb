"""The packed cluster engine (one vector S = |o> + |v> on an even lattice)
against the oracle: every split of the lattice into pencils that changes the
code path -- one CTA, pencils of one row, odd numbers of rows, 1 to 4 pairs of
sites per thread, threads left over -- at the smallest and larger M, with K = M
and K = 2M nodes.

Tolerances: FP64 Delta Omega 1e-10 |dO| + 1e-13 a; FP32-mixed 2e-5 t (the
tolerance of FP32 moments: 6e-8 rounding per step, M/2 steps, values <= 1).
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1303_6016_gb300 import inputs

pytestmark = pytest.mark.gpu

A = 6.05


@pytest.fixture(scope="module")
def G():
    from paper_1303_6016_gb300 import build, gfmc
    build.build()
    gfmc.load()
    return gfmc


def replay(L, sp, M, nodes, chain_id, out, tol, tie):
    n = out["decisions"].size
    res = O.updates(L, sp, n, M, beta=12.0, chem=-2.0, seed=5, chain_id=chain_id, nodes=nodes or None,
                    forced=out["decisions"].astype(np.int8))
    for q in range(n):
        assert abs(out["d_omega"][q] - res["d_omega"][q]) <= tol(res["d_omega"][q]), (L, q)
        if bool(res["ratio"][q] > res["u"][q]) != bool(out["decisions"][q]):
            assert abs(res["ratio"][q] - res["u"][q]) < tie


@pytest.mark.parametrize("precision,tol,tie", [
    ("fp64", lambda r: 1e-10 * abs(r) + 1e-13 * A, 1e-9),
    ("fp32_mixed", lambda r: 2e-5, 1e-3),
])
def test_packed_clusters_match_oracle(G, precision, tol, tie):
    # (L, CTAs, M, nodes): one CTA; pencils of one row (4, 4); odd row counts (6, 2), (10, 2),
    # (14, 2); 3 and 4 pairs per thread in FP32 (14, 1), (12, 1), (16, 2); FFT parts 1, 2 and 4
    specs = [(4, 1, 16, 0), (4, 2, 64, 128), (4, 4, 32, 0), (6, 1, 64, 0), (6, 2, 16, 32), (8, 8, 64, 0),
             (10, 2, 32, 64), (12, 1, 64, 0), (14, 2, 32, 0), (16, 2, 16, 0), (16, 16, 32, 64), (20, 4, 16, 0)]
    if precision == "fp32_mixed":
        specs += [(14, 1, 32, 0), (18, 2, 16, 0)]
    n = 24
    chains, sps = [], []
    for c, (L, _, M, nodes) in enumerate(specs):
        sps.append(inputs.uniform_sphere(L, 40 + c))
        chains.append(G.Chain(L, sps[c], M=M, beta=12.0, mu=-2.0, seed=5, chain_id=c, precision=precision,
                              recursion="proposal", nodes=nodes))
    outs = G.run_clusters(chains, n, [s[1] for s in specs])
    for c, (L, _, M, nodes) in enumerate(specs):
        replay(L, sps[c], M, nodes, c, outs[c], tol, tie)
    for ch in chains:
        ch.close()


@pytest.mark.parametrize("L,M,n", [(4, 64, 80), (6, 128, 12), (10, 64, 12), (14, 32, 12), (16, 64, 10), (18, 16, 10),
                                   (20, 32, 8), (24, 16, 8), (34, 16, 4), (48, 16, 3)])
def test_fp64_single_chains_match_oracle(G, L, M, n):
    """FP64 chains on the automatic engine, the fixed-point recursion: one
    cluster (parts of sites and whole sites per thread, a cluster of 6, 10 or 14
    CTAs) and the whole grid (pencils of one to sixteen rows, of unequal size,
    1 to 3 sites per thread), a full sweep with its magnetisation, Delta Omega of
    a given proposal, and a rerun bit for bit."""
    sp = inputs.von_mises_fisher(L, 2.0, L)
    kw = dict(M=M, beta=12.0, mu=-2.0, seed=5, chain_id=3)
    tol, tie = lambda r: 1e-10 * abs(r) + 1e-13 * A, 1e-9
    with G.Chain(L, sp, **kw) as ch:
        o = L ** 3 // 2 + 3
        d, ref = ch.delta_omega(o, 1.1, 2.3), O.delta_omega(L, sp, o, 1.1, 2.3, M, beta=12.0, chem=-2.0)
        assert abs(d - ref) <= tol(ref)
        out = ch.updates(n)
        replay(L, sp, M, 0, 3, out, tol, tie)
        assert out["magnetization"].size == n // L ** 3
    with G.Chain(L, sp, **kw) as ch:
        again = ch.updates(n)
    assert np.array_equal(again["d_omega"], out["d_omega"])


def test_packed_grid_wait_runs_out(G):
    """A chain on the whole grid whose CTA 0 sends no face values: the bounded
    waits of its neighbours end the launch with GFMC_ETIMEOUT, and the chain then
    runs on as if nothing had happened."""
    L, M, n = 20, 16, 6
    sp = inputs.uniform_sphere(L, 1)
    with G.Chain(L, sp, M=M, seed=3) as a, G.Chain(L, sp, M=M, seed=3) as b:
        a.set_wait_budget(20_000_000)
        a.inject_stall(True)
        with pytest.raises(G.GfmcError) as e:
            a.updates(n)
        assert e.value.status == G.GFMC_ETIMEOUT
        a.set_wait_budget(4_000_000_000)
        assert np.array_equal(a.updates(n)["d_omega"], b.updates(n)["d_omega"])


@pytest.mark.parametrize("precision,tol,tie", [
    ("fp64", lambda r: 1e-10 * abs(r) + 1e-13 * A, 1e-9),
    ("fp32_mixed", lambda r: 2e-5, 1e-3),
])
def test_teams_match_oracle(G, precision, tol, tie):
    """Chains on teams of CTAs, both recursions: one CTA of 1, 2, 3 and 4 sites per
    thread and more; tiles of a plane and more with the planes beside them in
    shared memory (the whole lattice, tiles all edge, tiles with an interior,
    tiles of unequal size) and tiles below a plane; odd lattices; chains on two
    and on seven vectors sharing a CTA.  nsteps of 7, 8, 9 and 15 around the
    groups of eight steps."""
    # (L, team size, M, recursion, engine)
    specs = [(4, 1, 16, "unit_vectors", "auto"), (6, 0, 32, "unit_vectors", "auto"),
             (5, 0, 16, "unit_vectors", "auto"), (6, 0, 16, "unit_vectors", "grid"),
             (8, 0, 16, "unit_vectors", "auto"), (8, 1, 64, "proposal", "auto"), (10, 1, 32, "unit_vectors", "auto"),
             (12, 1, 16, "proposal", "auto"), (4, 2, 32, "unit_vectors", "auto"), (6, 3, 32, "proposal", "auto"),
             (8, 3, 16, "unit_vectors", "auto"), (8, 20, 16, "unit_vectors", "auto"),
             (10, 7, 32, "proposal", "auto"), (12, 5, 16, "unit_vectors", "auto"),
             (14, 3, 32, "unit_vectors", "auto"), (7, 2, 16, "unit_vectors", "auto")]
    n = 14
    chains, sps = [], []
    for c, (L, _, M, rec, eng) in enumerate(specs):
        sps.append(inputs.uniform_sphere(L, 70 + c))
        chains.append(G.Chain(L, sps[c], M=M, beta=12.0, mu=-2.0, seed=5, chain_id=c, precision=precision,
                              recursion=rec, engine=eng))
    outs = G.run_batch(chains, n, team_ctas=[s[1] for s in specs])
    for c, (L, _, M, _, _) in enumerate(specs):
        replay(L, sps[c], M, 0, c, outs[c], tol, tie)
    for ch in chains:
        ch.close()


@pytest.mark.parametrize("L,M,nodes,n", [(4, 16, 0, 70), (4, 64, 128, 10), (6, 32, 0, 10), (8, 64, 0, 10),
                                         (10, 32, 64, 6)])
def test_fp32_single_chains_match_oracle(G, L, M, nodes, n):
    """FP32-mixed chains on the automatic engine: one CTA of fewer sites than threads, of
    a site per thread of 256 and of 512 threads, a full sweep at L = 4, and the first
    size on a cluster."""
    sp = inputs.von_mises_fisher(L, 2.0, L)
    with G.Chain(L, sp, M=M, beta=12.0, mu=-2.0, seed=5, chain_id=3, precision="fp32_mixed", nodes=nodes) as ch:
        out = ch.updates(n)
        replay(L, sp, M, nodes, 3, out, lambda r: 2e-5, 1e-3)
        assert out["magnetization"].size == n // L ** 3


@pytest.mark.parametrize("L,M", [(4, 16), (4, 64), (6, 64), (8, 32), (10, 32), (12, 16), (14, 16), (16, 64)])
@pytest.mark.parametrize("precision", ["fp64", "fp32_mixed"])
def test_moments_on_clusters_match_oracle(G, L, M, precision):
    """Moments read off six vectors on clusters: 1/4 of a site, half a site and a
    whole site per thread, sites on every face of the lattice.  Tolerance: 2^-60 per
    step and site, and the oracle's doubling, 1e-13 for values <= 1."""
    sp = inputs.von_mises_fisher(L, 2.0, L)
    with G.Chain(L, sp, M=M, precision=precision) as ch:
        for o in (0, L ** 3 - 1, L ** 3 // 2 + 3):
            mu = ch.moments(o)
            assert np.abs(mu - O.moments(L, sp, o, M)).max() <= 1e-13
            assert np.array_equal(mu, mu.transpose(1, 0, 2).conj())
        assert np.array_equal(mu, ch.moments(o))
