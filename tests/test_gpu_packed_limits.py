"""The packed engines beside the other calls of a chain, and where they end: a chain
in a batch and then alone, waits that run out on a cluster,
teams on as many nodes as the tail takes, teams beside other chains, and the sizes
at the far ends of the ranges, against the oracle."""
import time

import numpy as np
import pytest

from paper_1303_6016_gb300 import inputs
from test_gpu_packed import A, replay

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


def _times_out(G, ch, call):
    """A stalled call ends with GFMC_ETIMEOUT in little more than one budget of 10 ms."""
    ch.set_wait_budget(20_000_000)
    ch.inject_stall(True)
    t = time.perf_counter()
    with pytest.raises(G.GfmcError) as e:
        call()
    assert e.value.status == G.GFMC_ETIMEOUT
    assert time.perf_counter() - t < 1.0
    ch.set_wait_budget(4_000_000_000)


@pytest.mark.parametrize("L,M,n", [(8, 16, 300), (12, 64, 300), (16, 64, 300)])
def test_cluster_wait_runs_out(G, L, M, n):
    """An FP64 chain on one cluster (a quarter, half a site and a site per thread) whose CTA 0
    sends no face values: the waits of the others run out once and the launch ends,
    however many updates are left, and the chain runs on as if nothing had happened."""
    sp = inputs.uniform_sphere(L, 1)
    with G.Chain(L, sp, M=M, seed=3) as a, G.Chain(L, sp, M=M, seed=3) as b:
        _times_out(G, a, lambda: a.updates(n))
        assert a.counter == 0
        assert np.array_equal(a.updates(20)["d_omega"], b.updates(20)["d_omega"])
        _times_out(G, a, lambda: a.delta_omega(5, 1.0, 2.0))
        assert a.delta_omega(5, 1.0, 2.0) == b.delta_omega(5, 1.0, 2.0)


@pytest.mark.parametrize("L,M", [(4, 16), (8, 64), (16, 64)])
def test_moments_wait_runs_out(G, L, M):
    """The same on the six clusters of a moments call."""
    sp = inputs.uniform_sphere(L, 1)
    with G.Chain(L, sp, M=M) as ch:
        ref = ch.moments(7)
        _times_out(G, ch, lambda: ch.moments(7))
        assert np.array_equal(ch.moments(7), ref)


@pytest.mark.parametrize("small,large", [((8, 1), (24, 1)), ((6, 1), (8, 20))])
def test_team_batch_on_8192_nodes(G, small, large):
    """FP32 chains of M = 4096 on 2M nodes, whose tail alone takes 128 KB of a CTA's
    shared memory: one with its vectors there beside one whose vectors stay in global
    memory (a lattice too large, a tile below a plane) in one batch and in one plan, each
    as in a batch of its own."""
    specs = [small, large]
    sps = [inputs.uniform_sphere(L, 5 + c) for c, (L, _) in enumerate(specs)]

    def chains():
        return [G.Chain(L, sps[c], M=4096, nodes=8192, seed=2, chain_id=c, precision="fp32_mixed")
                for c, (L, _) in enumerate(specs)]

    ref = []
    for c, ch in enumerate(chains()):
        ref.append(G.run_batch([ch], 2, team_ctas=[specs[c][1]])[0]["d_omega"])
        ch.close()
    both = chains()
    for r, out in zip(ref, G.run_batch(both, 2, team_ctas=[tc for _, tc in specs])):
        assert np.array_equal(out["d_omega"], r)
    for ch in both:
        ch.close()
    both = chains()
    with G.Plan(both, 2, [tc for _, tc in specs], schedule="teams") as plan:
        plan.launch(1)
        for r, out in zip(ref, plan.sync()):
            assert np.array_equal(out["d_omega"], r)
    for ch in both:
        ch.close()


@pytest.mark.parametrize("precision,L,team,other", [
    ("fp32_mixed", 32, 3, dict(L=5)), ("fp32_mixed", 32, 3, dict(L=6, engine="grid")),
    ("fp32_mixed", 32, 4, dict(L=6, engine="grid")), ("fp32_mixed", 12, 1, dict(L=4, M=4096, nodes=8192)),
    ("fp32_mixed", 10, 1, dict(L=6, engine="grid", M=4096, nodes=8192)), ("fp64", 24, 8, dict(L=4, M=4096, nodes=8192)),
    ("fp64", 8, 1, dict(L=5, M=4096, nodes=8192))])
def test_team_results_do_not_depend_on_the_other_chains(G, precision, L, team, other):
    """A chain on a team whose vectors fit in shared memory beside some chains and not
    beside others (another kernel's static share, the tail of another chain): the same
    bits in both launches."""
    kw = dict(M=64, beta=12.0, mu=-2.0, seed=5, precision=precision)
    sp = inputs.uniform_sphere(L, 3)
    okw = {**kw, **{k: v for k, v in other.items() if k != "L"}}
    with G.Chain(L, sp, **kw) as a, G.Chain(L, sp, **kw) as b, \
            G.Chain(other["L"], inputs.uniform_sphere(other["L"], 4), **okw) as o:
        ra = G.run_batch([a], 3, team_ctas=[team])[0]
        rb = G.run_batch([b, o], 3, team_ctas=[team, 1])[0]
        assert np.array_equal(ra["d_omega"], rb["d_omega"])


@pytest.mark.parametrize("L,teams", [(12, (1, 2, 5, 20)), (16, (1, 3, 8, 20)), (24, (3, 20))])
def test_fp32_team_sums_do_not_depend_on_the_tiles(G, L, teams):
    """The products of an FP32 chain's steps are summed as integers, site by site, so that
    Delta Omega is the same on one CTA, on tiles of planes with and without an interior, of
    unequal size, and on tiles below a plane -- to the FP64 additions of the tail's phase sum,
    which is cut over the CTAs: K = 64 terms of a sum of order 1, 64 x 2^-53 < 1e-14 (sums in
    FP32 differ by 1e-8)."""
    sp = inputs.von_mises_fisher(L, 5.0, 3)
    chains = [G.Chain(L, sp, M=64, beta=12.0, mu=-2.0, seed=5, precision="fp32_mixed") for _ in teams]
    outs = [G.run_batch([ch], 4, team_ctas=[tc])[0]["d_omega"] for ch, tc in zip(chains, teams)]
    for o in outs[1:]:
        assert np.abs(o - outs[0]).max() <= 1e-14
    for ch in chains:
        ch.close()


@pytest.mark.parametrize("L,M,n", [(50, 16, 2), (62, 16, 1), (64, 16, 1)])
def test_large_fp64_single_chains_match_oracle(G, L, M, n):
    """FP64 chains alone beyond three sites per thread of the whole grid (bonds and S_{m-1} from
    shared memory, up to six face values per thread: L = 50 to 62), and L = 64, which the
    grid does not hold: the team engine on two vectors.  Tolerance as in test_gpu_packed."""
    sp = inputs.von_mises_fisher(L, 2.0, L)
    with G.Chain(L, sp, M=M, beta=12.0, mu=-2.0, seed=5, chain_id=3) as ch:
        out = ch.updates(n)
    replay(L, sp, M, 0, 3, out, lambda r: 1e-10 * abs(r) + 1e-13 * A, 1e-9)


@pytest.mark.parametrize("L,M,nodes,n", [(14, 32, 0, 8), (20, 16, 0, 6), (22, 16, 0, 4), (26, 16, 32, 3),
                                         (30, 16, 0, 2), (40, 16, 0, 2), (34, 16, 0, 2)])
def test_larger_fp32_single_chains_match_oracle(G, L, M, nodes, n):
    """FP32-mixed chains alone on a cluster, of 14, 16, 11 (cut along z alone), 13, 15 and 16
    CTAs, with one, two and four pairs of sites per thread; and L = 34, which no cluster
    takes."""
    sp = inputs.von_mises_fisher(L, 2.0, L)
    with G.Chain(L, sp, M=M, beta=12.0, mu=-2.0, seed=5, chain_id=3, precision="fp32_mixed", nodes=nodes) as ch:
        out = ch.updates(n)
    replay(L, sp, M, nodes, 3, out, lambda r: 2e-5, 1e-3)


@pytest.mark.parametrize("L,C", [(12, 1), (24, 8)])
def test_fp64_clusters_on_8192_nodes_match_oracle(G, L, C):
    """The two sizes whose tail's 128 KB leave no room for a record per site, so that they run
    pk64_steps (everything in shared memory).  Tolerance: the oracle's FP64 rounding over M = 4096
    steps, 4096 x 2^-53 x a = 2.7e-12, taken four times."""
    M, n = 4096, 2
    sp = inputs.uniform_sphere(L, 9)
    with G.Chain(L, sp, M=M, nodes=8192, beta=12.0, mu=-2.0, seed=5, chain_id=3, recursion="proposal") as ch:
        out = G.run_clusters([ch], n, [C])[0]
    replay(L, sp, M, 8192, 3, out, lambda r: 1.1e-11, 1e-9)
