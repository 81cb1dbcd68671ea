"""An RVE's FP64 result is the same bits whatever shares its batch: a batch of few
RVEs divides each over more CTAs than a full one (fp64_parts.h), and the sums go by
groups of nodes that do not depend on it."""
import numpy as np
import pytest

import rve_inputs as ri

pytestmark = pytest.mark.gpu

ITERS = 50


def _solve(nets, F, c, block):
    from paper_2305_07030_gb300 import Batch
    with Batch(nets, damping=c) as b:
        b.solve(F, precision="fp64", init="affine", tol=0.0, max_iter=ITERS, kinetic_energy=True, block_threads=block)
        kinetic = b.diagnostics()["kinetic_energy"][0]  # summed at the end of the solve
        b.solve(F, precision="fp64", init="affine", tol=0.0, max_iter=ITERS, kinetic_energy="balance",
                block_threads=block)
        out, e = b.stress(), b.energy()
        res = {k: out[k][0] for k in ("sigma", "iters", "rel_res")}
        res.update({k: v[0] for k, v in e.items()}, f_ref=b.diagnostics()["f_ref"][0])
        assert kinetic == e["kinetic"][0]  # with the energy check in every iteration
        return res, b.displacement()[:nets[0].n_nodes]


# one group, 2 to 16 groups of one mixed part, several mixed parts; parts whose state
# (16 of 1125 nodes) and tables (of 1250 and 2100) do not fit in shared memory
@pytest.mark.parametrize("n", [60, 80, 200, 512, 700, 1500, 2600, 5000, 18000, 20000, 33000])
def test_alone_equals_among_others(n):
    rng = np.random.default_rng(n)
    net, tiny = ri.random_network(n, rng), ri.random_network(37, rng)
    F, c = ri.symmetric_perturbation(rng), ri.default_damping(n)
    one, u = _solve([net], F[None], [c], 0)
    # companions that leave room for every split, for smaller ones and for none; CTA sizes
    for others, block in ((6, 0), (20, 0), (50, 0), (130, 0), (0, 64), (130, 256)):
        got, v = _solve([net] + [tiny] * others, np.repeat(F[None], others + 1, axis=0),
                        [c] + [ri.default_damping(37)] * others, block)
        assert np.array_equal(u, v), (others, block)
        for k, x in one.items():
            assert np.array_equal(x, got[k]), (others, block, k)
