"""FP64 on more CTAs than the mixed solver's parts: small batches are split further
(runtime.cu, fp64_split), and the allocation-free call splits its nodes itself
(noalloc.cu). The trajectory stays the oracle's bit for bit, whatever the split."""
import numpy as np
import pytest

import oracle
import rve_inputs as ri

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

ITERS = 60


def _net(n, seed):
    rng = np.random.default_rng(seed)
    net = ri.random_network(n, rng)
    return net, ri.symmetric_perturbation(rng), ri.default_damping(n)


# below and at 2, 4, 8 and 16 parts of 40 nodes, several mixed parts, and the
# allocation-free call's largest RVE
@pytest.mark.parametrize("n", [12, 37, 79, 80, 159, 160, 319, 320, 639, 640, 700, 1500, 2600, 4096])
def test_bitwise_against_oracle(n):
    import paper_2305_07030_gb300 as fe2
    net, F, c = _net(n, n)
    ref = oracle.solve_batch(ri.Workload("split", [net], F[None], np.array([c])), init=1, tol=0.0, max_iter=ITERS)[0]
    with fe2.Batch([net], damping=[c]) as b:
        b.solve(F[None], precision="fp64", init="affine", tol=0.0, max_iter=ITERS)
        out, u = b.stress(), b.displacement()
    assert out["iters"][0] == ref["iters"] and np.array_equal(u, ref["u"])
    assert abs(out["rel_res"][0] - ref["rel_res"]) <= 1e-12 * ref["rel_res"]

    def dev(a):
        return torch.as_tensor(np.ascontiguousarray(a), device="cuda")

    un = torch.zeros(n, 3, dtype=torch.float64, device="cuda")
    sig = torch.zeros(3, 3, dtype=torch.float64, device="cuda")
    it = torch.zeros(1, dtype=torch.int64, device="cuda")
    rr = torch.zeros(1, dtype=torch.float64, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    fe2.rve_solve_noalloc(n, len(net.elems), dev(net.X), dev(net.elems), dev(net.EA), dev(net.fixed), dev(F), un, sig,
                          it, rr, st, damping=c, stream=torch.cuda.current_stream(), precision="fp64", init="affine",
                          tol=0.0, max_iter=ITERS)
    torch.cuda.synchronize()
    assert int(it) == ref["iters"] and np.array_equal(un.cpu().numpy(), ref["u"])
    assert abs(float(rr) - ref["rel_res"]) <= 1e-12 * ref["rel_res"]
    assert np.abs(sig.cpu().numpy() - ref["sigma"]).max() <= 1e-12 * np.abs(ref["sigma"]).max()


def test_split_and_whole_rves_agree():
    """The same RVE in a batch that fills the GPU (its own parts) and alone (split):
    equal displacements, and energies and residuals up to the order of their sums."""
    import paper_2305_07030_gb300 as fe2
    net, F, c = _net(700, 5)
    opts = dict(precision="fp64", init="affine", tol=0.0, max_iter=ITERS, kinetic_energy="balance")
    with fe2.Batch([net], damping=[c]) as b:
        b.solve(F[None], **opts)
        one, u, e1 = b.stress(), b.displacement(), b.energy()
    with fe2.Batch([net] * 200, damping=[c] * 200) as b:
        b.solve(np.repeat(F[None], 200, axis=0), **opts)
        many, v, e2 = b.stress(), b.displacement(), b.energy()
    for p in range(200):
        assert np.array_equal(u, v[700 * p:700 * (p + 1)])
    assert np.array_equal(one["sigma"][0], many["sigma"][0]) and one["iters"][0] == many["iters"][0]
    assert abs(one["rel_res"][0] - many["rel_res"][0]) <= 1e-12 * one["rel_res"][0]
    for k in ("kinetic", "internal_work", "external_work"):
        assert abs(e1[k][0] - e2[k][0]) <= 1e-10 * max(abs(e1["kinetic"][0]), abs(e1["internal_work"][0]))
