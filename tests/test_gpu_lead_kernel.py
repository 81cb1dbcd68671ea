"""The lead kernel (csrc/dr_mixed_lead.cu): double-float iterations against the FP64
oracle at the edges of its variants, and the same bits whatever the CTA size."""
import numpy as np
import pytest

import oracle
import rve_inputs as ri

pytestmark = pytest.mark.gpu

ITERS = 40
# Double-float operations are good to 2^-44; an error in the velocity is carried
# on over the remaining iterations (ITERS^2 / 2), about 8 operations each, and the
# networks' unstable directions may raise it another 16 times.
TOL = ITERS ** 2 / 2 * 8 * 16 * 2.0 ** -44


def _graph(n, rng):
    """Elements between random nodes: almost every node has neighbours in almost
    every part."""
    base = ri.random_network(n, rng)
    e = np.sort(rng.integers(0, n, (3 * n, 2)), axis=1)
    e = np.unique(e[e[:, 0] != e[:, 1]], axis=0).astype(np.int32)
    return ri.Network(X=base.X, elems=e, EA=rng.lognormal(0.0, 0.3, len(e)), fixed=base.fixed)


# A handful of free nodes; one part with and without the shared element table (700
# and 790 nodes); 2, 8 and 16 parts; parts without the table (13,000 and 33,000
# nodes); element constants in global memory and no table kernel at all (graphs).
@pytest.mark.parametrize("kind,n", [("net", n) for n in (37, 60, 512, 700, 790, 1500, 5000, 13000, 33000)] +
                         [("graph", 1500), ("graph", 3000), ("graph", 9000)])
@pytest.mark.parametrize("init", ["affine", "reference"])
def test_lead_against_oracle(kind, n, init):
    from paper_2305_07030_gb300 import Batch
    rng = np.random.default_rng(n)
    net = _graph(n, rng) if kind == "graph" else ri.random_network(n, rng)
    F = np.array([ri.symmetric_perturbation(rng)])
    if init == "reference":
        F = np.eye(3) + 0.05 * (F - np.eye(3))  # small: the first steps stay smooth
    c = np.array([ri.default_damping(n)])
    ref = oracle.solve_batch(ri.Workload("lead", [net], F, c), init=1 if init == "affine" else 0, tol=0.0,
                             max_iter=ITERS)[0]
    move = np.abs(ref["u"]).max()
    first = None
    for block in (0, 64, 160, 256):
        with Batch([net], damping=c) as b:
            b.solve(F, precision="mixed", init=init, tol=0.0, max_iter=ITERS, lead_iters=ITERS, block_threads=block)
            out, u = b.stress(), b.displacement()
        assert out["iters"][0] == ITERS
        assert np.abs(u - ref["u"]).max() <= TOL * move
        if first is None:
            first = u
        assert np.array_equal(u, first), block
