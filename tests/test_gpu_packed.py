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
