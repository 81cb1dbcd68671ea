"""The mixed solver's table kernels. The FP32 phase's (csrc/dr_mixed_node.cu): its
variants (one slab per warp in registers, several slabs, two CTAs per SM, tables
partly in global memory) run the same arithmetic, so the displacement does not
depend on the variant, the CTA size or the other RVEs of the launch. The lead's
(csrc/dr_mixed_lead.cu): likewise, and against the oracle."""
import numpy as np
import pytest

import rve_inputs as ri
from parity_util import check_equilibrium, rel_err

pytestmark = pytest.mark.gpu

LEAD, ITERS = 4, 44


def _nets(sizes, seed):
    rng = np.random.default_rng(seed)
    nets = [ri.random_network(int(n), rng) for n in sizes]
    F = np.array([ri.symmetric_perturbation(rng) for _ in nets])
    c = np.array([ri.default_damping(n.n_nodes) for n in nets])
    return nets, F, c


def _solve(nets, F, c, **kw):
    from paper_2305_07030_gb300 import Batch
    with Batch(nets, damping=c) as b:
        b.solve(F, precision="mixed", init="affine", tol=0.0, max_iter=ITERS, lead_iters=LEAD, **kw)
        out = b.stress()
        return dict(out, f_ref=b.diagnostics()["f_ref"]), b.displacement(), b.node_off


def _state_is_the_tested_one(net, F, u, out, p):
    """The reported residual and stress are those of the returned displacement
    by the oracle's force law: the solve ends with the evaluation it tested. A
    nodal force is a double-float sum plus at most a dozen FP32 increments of
    relative error 16 x 2^-24, each up to about 100 times the net force: 1e-3
    with room."""
    res, sigma = check_equilibrium(net, F, u, out["f_ref"][p], 1e-8)
    assert out["iters"][p] == ITERS
    assert abs(res - out["rel_res"][p]) <= 1e-3 * res
    assert rel_err(out["sigma"][p], sigma) <= 1e-12


# Sizes around the tile edges: a handful of free nodes, slabs of 32, parts of
# about 512 free nodes (one slab per warp or two), 2, 4, 8 and 16 parts, parts
# whose tables exceed shared memory (33,000 nodes).
@pytest.mark.parametrize("n", [37, 60, 512, 700, 712, 1500, 2600, 5000, 11500, 13000, 33000])
def test_variants_agree(n):
    nets, F, c = _nets([n], seed=n)
    base, u, _ = _solve(nets, F, c)
    _state_is_the_tested_one(nets[0], F[0], u, base, 0)
    for block in (64, 160, 320):
        out, v, _ = _solve(nets, F, c, block_threads=block)
        assert np.array_equal(u, v), block
        # only the order of the residual's sum differs
        assert abs(out["rel_res"][0] - base["rel_res"][0]) <= 2.0 ** -20 * base["rel_res"][0]


@pytest.mark.parametrize("every", [1, 2, 3, 4, 5, 13])
def test_reference_refreshes(every):
    """Refreshes after a few evaluations test every pending evaluation first."""
    nets, F, c = _nets([300, 1500, 5000], seed=7)
    out, u, off = _solve(nets, F, c, rebase_every=every)
    for p, net in enumerate(nets):
        _state_is_the_tested_one(net, F[p], u[off[p]:off[p + 1]], out, p)


@pytest.mark.parametrize("n,copies", [(512, 160), (1000, 80), (5000, 20)])
def test_two_ctas_per_sm_match_one(n, copies):
    """More RVEs than one CTA per SM holds: each as when solved alone."""
    nets, F, c = _nets([n], seed=n + 1)
    one, u, _ = _solve(nets, F, c)
    out, v, off = _solve(nets * copies, np.repeat(F, copies, axis=0), np.repeat(c, copies))
    for p in range(copies):
        assert np.array_equal(u, v[off[p]:off[p + 1]])
        assert np.array_equal(one["sigma"][0], out["sigma"][p]) and one["rel_res"][0] == out["rel_res"][p]
