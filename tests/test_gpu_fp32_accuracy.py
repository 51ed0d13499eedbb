"""Accuracy of FP32-mixed Delta Omega on the packed recursion, against FP64 chains (in
fixed point, 1e-14): no worse than the two vectors one after the other on the grid engine
(engine "grid", plain sums), whose steps form the bond sum first and add a warp's
products in FP32 and the warps' in FP64.

Bound: the errors are the vectors' and the sums' rounding; the first alike, the second
smaller, so the ratio of the rms errors is 1 or below, and 1.1 passes (everything here is
deterministic).  Steps that add the bonds onto the older vector, so that every term rounds
at its magnitude, and sums of a warp or a tile in FP32 give 1.15 to 1.4."""
import numpy as np
import pytest

from paper_1303_6016_gb300 import inputs

pytestmark = pytest.mark.gpu

M, CHAINS, UPDATES = 256, 12, 6
SIZES = (12, 16, 24)


@pytest.fixture(scope="module")
def G():
    from paper_1303_6016_gb300 import build, gfmc
    build.build()
    gfmc.load()
    return gfmc


def run(G, L, how, ctas=None, **kw):
    """Delta Omega and decisions of CHAINS chains, [CHAINS][UPDATES]."""
    chains = [G.Chain(L, inputs.uniform_sphere(L, 300 + c), M=M, beta=20.0, mu=-2.0, seed=7, chain_id=c, **kw)
              for c in range(CHAINS)]
    if how == "cluster":
        outs = G.run_clusters(chains, UPDATES, [ctas] * CHAINS)
    elif how == "team":
        outs = G.run_batch(chains, UPDATES, team_ctas=[ctas] * CHAINS)
    else:
        outs = [ch.updates(UPDATES) for ch in chains]
    for ch in chains:
        ch.close()
    return [o["d_omega"] for o in outs], [o["decisions"] for o in outs]


def squares(G, L, exact, how, ctas=None, **kw):
    """Squared errors of the updates up to the first that decided otherwise."""
    dom, dec = run(G, L, how, ctas, precision="fp32_mixed", **kw)
    out = []
    for d, e, x, y in zip(dom, dec, *exact):
        for q in range(UPDATES):
            out.append((d[q] - x[q]) ** 2)
            if e[q] != y[q]:
                break
    return out


@pytest.fixture(scope="module")
def reference(G):
    exact = {L: run(G, L, "single") for L in SIZES}
    two = []
    for L in SIZES:
        two += squares(G, L, exact[L], "single", engine="grid", recursion="proposal")
    return exact, np.sqrt(np.mean(two))


@pytest.mark.parametrize("how,ctas", [("single", {}), ("cluster", {12: 1, 16: 2, 24: 8}), ("team", {12: 1, 16: 2, 24: 4})])
def test_packed_fp32_is_as_exact_as_two_vectors(G, reference, how, ctas):
    exact, two = reference
    kw = dict(recursion="proposal") if how == "cluster" else {}
    err = []
    for L in SIZES:
        err += squares(G, L, exact[L], how, ctas.get(L), **kw)
    assert np.sqrt(np.mean(err)) <= 1.1 * two


def test_one_cta_fp32_is_as_exact_as_seven_vectors(G):
    """Sizes that one CTA takes with its sites in registers, alone (a site per thread) and as
    a team of one CTA (two): threads' sums added as integers, so no worse than the seven
    unit vectors on the grid engine (sums of a warp in FP32: 1.06 of them, so 0.65)."""
    exact = run(G, 8, "single")
    seven = squares(G, 8, exact, "single", engine="grid")
    for how, ctas in (("single", None), ("team", 1)):
        assert np.mean(squares(G, 8, exact, how, ctas)) <= np.mean(seven)


@pytest.mark.parametrize("L", [6, 8, 10, 16, 34])
@pytest.mark.parametrize("move", [1e-1, 1e-3, 1e-5])
def test_small_moves(G, L, move):
    """A proposal close to the spin: FP32-mixed Delta Omega, of the order of the move, keeps the
    relative accuracy of a large one, on one CTA, clusters and tiles -- the sums' integers of
    2^-41 resolve a small v only because it is scaled.  Bound: 2e-5 for Delta Omega of order 1
    (the tolerance of FP32 moments), so 2e-5 of the move; and 1e-4 of Delta Omega itself."""
    sp = inputs.uniform_sphere(L, 21)
    o = L ** 3 // 2 + 1
    th = sp[o, 0] + (0.6 if sp[o, 0] < 1.5 else -0.6) * move
    ph = sp[o, 1] + 0.8 * move
    kw = dict(M=128, beta=12.0, mu=-2.0)
    with G.Chain(L, sp, **kw) as a, G.Chain(L, sp, precision="fp32_mixed", **kw) as b:
        d64, d32 = a.delta_omega(o, th, ph), b.delta_omega(o, th, ph)
    assert abs(d32 - d64) <= 2e-5 * move
    assert abs(d32 - d64) <= 1e-4 * abs(d64)
