"""Networks that connect almost every part with every other: the mixed solver's less
common routes, chosen by what fits in shared memory. The host-only plan says which
route a network takes, and on a GPU each one is run: the kernels without tables
(csrc/dr_mixed.cu), the lead with its element constants in global memory, and the
stall hand-back between them."""
import numpy as np
import pytest

import oracle
import rve_inputs as ri
from parity_util import check_equilibrium, rel_err

SMEM_OPTIN = 232448  # GB300 opt-in shared memory per block
LIMIT = SMEM_OPTIN - 16384
ITERS = 40

# (nodes, mean degree): lead, FP32 phase. "plain": without tables; "constants":
# all constants in shared memory; "no constants": only displacements and forces.
ROUTES = {(1600, 6): ("constants", "tables"), (3600, 6): ("no constants", "tables"),
          (4000, 6): ("constants", "tables"), (1600, 10): ("no constants", "tables"),
          (9000, 10): ("plain", "tables"), (20000, 6): ("plain", "plain"), (2500, 1200): ("plain", "plain")}


def _graph(n, deg):
    rng = np.random.default_rng(n)
    base = ri.random_network(n, rng)
    e = np.sort(rng.integers(0, n, (deg * n // 2, 2)), axis=1)
    e = np.unique(e[e[:, 0] != e[:, 1]], axis=0).astype(np.int32)
    return ri.Network(X=base.X, elems=e, EA=rng.lognormal(0.0, 0.3, len(e)), fixed=base.fixed)


def _displacements(net, L):
    """Most entries of a part's displacement array in the lead: its free nodes, one
    entry more, the free neighbours in other parts and the fixed neighbours."""
    C, perm = int(L["parts"][0]), L["perm"]
    pf = L["part_off"][0, 0]
    part = np.full(net.n_nodes, -1)
    for r in range(C):
        part[perm[pf[r]:pf[r + 1]]] = r
    a, b = net.elems.T
    most = 0
    for r in range(C):
        near = np.unique(np.concatenate([b[part[a] == r], a[part[b] == r]]))
        most = max(most, int(pf[r + 1] - pf[r]) + 1 + int((part[near] != r).sum()))
    return most


def _route(net):
    import paper_2305_07030_gb300 as m
    P, T = m.plan([net], smem_optin=SMEM_OPTIN), m.fp64_slots([net], smem_optin=SMEM_OPTIN)
    part = -(-net.n_nodes // int(P["parts"][0]))
    lead, fp32 = (int(x) for x in P["smem"][0])
    assert max(lead, fp32) <= LIMIT
    # displacements (two arrays in the staged form) and the slots' forces are 24 bytes
    # each, a slot's constants 44 more
    slots = int(np.diff(T["part_slot"][0]).max())
    base = 24 * ((2 if P["staged"][0, 0] else 1) * _displacements(net, m.layout([net], smem_optin=SMEM_OPTIN)) + slots)
    a = "plain" if lead == 32 * part else "constants" if lead >= base + 44 * slots else "no constants"
    assert a == "plain" or lead >= base
    return a, "plain" if fp32 == 96 * part else "tables"


@pytest.mark.parametrize("n,deg", list(ROUTES))
def test_route(n, deg):
    assert _route(_graph(n, deg)) == ROUTES[n, deg]


def _run(net, F, c, **kw):
    from paper_2305_07030_gb300 import Batch
    with Batch([net], damping=c) as b:
        b.solve(F, precision="mixed", init="affine", tol=0.0, **kw)
        return dict(b.stress(), **b.diagnostics()), b.displacement()


@pytest.mark.gpu
@pytest.mark.parametrize("n,deg", list(ROUTES))
def test_lead_against_oracle(n, deg):
    """Double-float operations are good to 2^-44; an error in the velocity is carried
    on over the remaining iterations (ITERS^2 / 2), about 8 operations each, the
    networks' unstable directions may raise it another 16 times, and a row's sum has
    as many terms as the node's degree (6 in the figure of 8)."""
    net, rng = _graph(n, deg), np.random.default_rng(n + 1)
    F, c = ri.symmetric_perturbation(rng)[None], np.array([ri.default_damping(n)])
    ref = oracle.solve_batch(ri.Workload("routes", [net], F, c), init=1, tol=0.0, max_iter=ITERS)[0]
    tol = ITERS ** 2 / 2 * 8 * 16 * max(1, deg / 6) * 2.0 ** -44
    for block in (0, 64, 160):
        out, u = _run(net, F, c, max_iter=ITERS, lead_iters=ITERS, block_threads=block)
        assert out["iters"][0] == ITERS and out["status"][0] == "MAXITER"
        assert np.abs(u - ref["u"]).max() <= tol * np.abs(ref["u"]).max()
        assert rel_err(out["sigma"][0], ref["sigma"]) <= tol


@pytest.mark.gpu
@pytest.mark.parametrize("n,deg", list(ROUTES))
@pytest.mark.parametrize("every,stall", [(0, 0), (7, 0), (0, 1)])
def test_fp32_phase_ends_with_the_tested_state(n, deg, every, stall):
    """The reported residual and stress are those of the returned displacement by the
    oracle's force law, also with refreshes of the reference and after a hand-back.
    A nodal force is a double-float sum plus its row's FP32 increments of relative
    error 16 x 2^-24, each up to about 100 times the net force: 1e-3 with room for a
    dozen of them, in proportion for longer rows."""
    net, rng = _graph(n, deg), np.random.default_rng(n + 1)
    F, c = ri.symmetric_perturbation(rng)[None], np.array([ri.default_damping(n)])
    out, u = _run(net, F, c, max_iter=ITERS, lead_iters=4, rebase_every=every, stall_window=stall)
    res, sigma = check_equilibrium(net, F[0], u, out["f_ref"][0], 1e-8)
    assert out["iters"][0] == ITERS
    assert abs(res - out["rel_res"][0]) <= 1e-3 * max(1, deg / 12) * res
    assert rel_err(out["sigma"][0], sigma) <= 1e-12
    # a hand-back after one evaluation leaves all but a few iterations to double-float
    assert out["lead_iters"][0] >= ITERS - 8 if stall else out["lead_iters"][0] == 4
