"""The FP32 phase's choice between one and two CTAs per SM (runtime.cu, pair_clusters)
goes by the iterations of the last mixed solve, and each choice has a CUDA graph of
its own: solve after solve on one batch gives the same bits, whatever the choice and
the order of the options."""
import numpy as np
import pytest

import rve_inputs as ri

pytestmark = pytest.mark.gpu


def test_repeated_solves_on_one_batch():
    from paper_2305_07030_gb300 import Batch
    rng = np.random.default_rng(3)
    net = ri.random_network(300, rng)
    P = 200  # more than one CTA per SM
    F = np.repeat(np.eye(3)[None], P, axis=0)
    F[7] = ri.symmetric_perturbation(rng)  # the one RVE that iterates
    every = np.repeat(F[7:8], P, axis=0)
    whole = dict(precision="mixed", init="affine", tol=1e-6, max_iter=200000)
    capped = dict(precision="mixed", init="affine", tol=0.0, max_iter=60, lead_iters=6)
    steps = [("slow", F, whole), ("slow", F, whole), ("even", every, capped), ("even", every, capped),
             ("slow", F, whole), ("fp64", F, dict(precision="fp64", tol=0.0, max_iter=20)), ("slow", F, whole),
             ("even", every, capped), ("slow", F, whole), ("slow", F, dict(whole, launch="stream"))]
    seen = {}
    with Batch([net] * P, damping=[ri.default_damping(300)] * P) as b:
        for name, f, opts in steps:
            b.solve(f, **opts)
            out = b.stress()
            got = [out["iters"], out["sigma"], out["rel_res"], b.displacement()]
            for x, y in zip(seen.setdefault(name, got), got):
                assert np.array_equal(x, y), name
    assert seen["slow"][0][7] > 100 * np.delete(seen["slow"][0], 7).max()
    # the RVE among its copies and alone
    assert np.array_equal(seen["even"][1][0], seen["even"][1][P - 1])
