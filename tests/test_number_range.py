"""Networks whose lengths or rigidities are near FP32's limits run the mixed solver's
table kernels like any other (csrc/dr_mixed_node.cu, without the flush to zero), and
scaling by a power of two scales their solution exactly."""
import numpy as np
import pytest

import rve_inputs as ri

# lengths beyond 1e6, rigidities beyond 1e15 and below 1e-15: outside the range in
# which the flushing forms are taken (runtime.cu, node_range_ok). The factors keep
# every product of the iterations normal, so the scaling is exact; with the last one
# the square of a small nodal force may be subnormal, which only the residual sees.
SCALES = [(2.0 ** 41, 1.0), (1.0, 2.0 ** 51), (1.0, 2.0 ** -51)]


def _net(n, length=1.0, rigidity=1.0):
    b = ri.random_network(n, np.random.default_rng(n))
    return ri.Network(X=b.X * length, elems=b.elems, EA=b.EA * rigidity, fixed=b.fixed, V0=length ** 3)


@pytest.mark.parametrize("length,rigidity", SCALES + [(1e-13, 1.0)])
def test_same_launch_plan(length, rigidity):
    from paper_2305_07030_gb300 import plan
    for n in (60, 700, 5000, 13000):
        a, b = plan([_net(n)]), plan([_net(n, length, rigidity)])
        for k in ("parts", "staged", "block", "smem"):
            assert np.array_equal(a[k], b[k]), (n, k)


# one part in registers, several slabs per warp, several parts, the other order of
# fused operations (13,000 nodes), rows in global memory (33,000)
@pytest.mark.gpu
@pytest.mark.parametrize("n", [60, 700, 1000, 5000, 13000, 33000])
def test_scaled_solution_is_exact(n):
    from paper_2305_07030_gb300 import Batch
    rng = np.random.default_rng(n + 1)
    F, c = ri.symmetric_perturbation(rng)[None], [ri.default_damping(n)]
    out = []
    for length, rigidity in [(1.0, 1.0)] + SCALES:
        with Batch([_net(n, length, rigidity)], damping=c) as b:
            b.solve(F, precision="mixed", init="affine", tol=0.0, max_iter=44, lead_iters=4, rebase_every=13)
            r, u = b.stress(), b.displacement()
        out.append((u / length, r["sigma"] * length ** 2 / rigidity, r["rel_res"], r["iters"]))
    for k, got in enumerate(out[1:]):
        for name, x, y in zip(("u", "sigma", "rel_res", "iters"), out[0], got):
            if name == "rel_res" and k == 2:
                assert abs(x - y) <= 2.0 ** -20 * x
            else:
                assert np.array_equal(x, y), (SCALES[k], name)
