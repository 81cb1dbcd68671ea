"""Shared-memory capacities of the mixed kernels (host-only plan, no GPU needed)."""
import numpy as np

import rve_inputs as ri


def test_parts_without_free_nodes_take_no_room():
    """A bar held fixed over one half: parts without free nodes have no copies in
    other parts, whichever end of the bar (and of the part order) they are at."""
    import paper_2305_07030_gb300 as m
    b = ri.random_network(3000, np.random.default_rng(5))
    X = b.X * np.array([8.0, 1.0, 1.0])
    fixed = ((X[:, 0] > 4.0) | (b.fixed != 0)).astype(np.uint8)
    plans = []
    for x in (X[:, 0], 8.0 - X[:, 0]):
        net = ri.Network(X=np.column_stack([x, X[:, 1:]]), elems=b.elems, EA=b.EA, fixed=fixed)
        pf = m.layout([net])["part_off"][0, 0, :5]
        assert np.diff(pf).min() == 0 and pf[4] > 0
        plans.append(m.plan([net]))
    assert plans[0]["parts"].tolist() == plans[1]["parts"].tolist() == [4]
    assert plans[0]["smem"].tolist() == plans[1]["smem"].tolist()
