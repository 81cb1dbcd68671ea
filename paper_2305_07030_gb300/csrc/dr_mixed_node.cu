// FP32 phase of the mixed solver: increment iterations of one RVE on a
// thread-block cluster, one thread per free node.
//
// What bounds it: instruction issue and the shared-memory pipe (an entry takes
// 11 to 16 wavefronts, 10 of them the random 16-byte gather of the neighbour's
// increment) while SMs are full, latency (the cluster barrier, about 1300 cycles
// for 8 CTAs, and the force chains) while they are not. Measured against the
// element-table kernel it replaced (each element once into a shared table, a CTA
// barrier, node sums), per iteration: 512 nodes on one CTA 2.2 -> 1.2 us, 5000
// nodes on 8 CTAs 2.5 -> 1.7 us, or 2.05 us with two CTAs on each SM; 20,000
// nodes on 16 CTAs, which had no tables, 7.9 -> 3.7 us.
//
// Arithmetic. Each element force is an exact increment about a reference state
// x_ref (dr_mixed.cu's header gives the formulas): every FP32 operation acts
// on small quantities, and the nodal sums of the reference forces (g_ref) are
// evaluated in double-float every rebase_every iterations, when the increment
// is folded into the double-float displacement.
//
// Layout. A node's owner thread evaluates the forces of its own row, in row
// order, and moves its node: nothing but the displacement increments passes
// between threads, so an iteration is one pass and one cluster barrier. Both
// ends of an element evaluate it, with exactly opposite results (r and dd
// change sign together, every other term is even in them).
//  * Rows are ELL-style slabs of 32 nodes: entry j of node k sits at slot
//    SS[k / 32] + 32 j + k % 32 and holds r = x_ref,j - x_ref,k, EA, q_ref and
//    the neighbour's place in the increment array. The free nodes of a part are
//    sorted by degree, so slabs have little padding; a padded entry is
//    the node itself with EA = q_ref = 0 and adds zero.
//  * The increment array of a CTA holds its own free nodes, one zero entry that
//    stands for every fixed node, and a copy of each free neighbour in another
//    CTA. The owner writes the copies (st.shared::cluster) when it moves its
//    node, so the barrier that makes them visible is the only wait, and the
//    force loop reads its own shared memory only. Two arrays alternate; the own
//    increments of the last four evaluations also go to a ring in global memory
//    (L2), written at the start of an iteration so that the barrier never
//    waits for them.
//  * Entries that do not fit in shared memory (parts of more than about 1000
//    nodes) are streamed from global memory (L2), whole slabs at a time.
//
// Residual test. Each thread leaves its squared residual in shared memory; while
// the next evaluation runs, the last warp adds them (FP32 per warp, the tree of a
// butterfly; double-float over the warps) and sends the sum to every CTA, totals
// the evaluation of three iterations back, and leaves a verdict that every warp
// reads after the next barrier.
#include <algorithm>
#include <map>
#include <mutex>
#include <utility>

#include "dr_mixed.cuh"

namespace fe2 {

namespace {

constexpr int kThreads = 512;
constexpr int kRing = 4;       // evaluations whose increments are kept
constexpr int kRegEntries = 6;  // row entries a thread keeps in registers (ONE)

struct NodeShared : ResidualSums {
    Verdict vd[2];                      // by evaluation parity
    double sig[kMaxParts][9];           // stress partials, read by rank 0
    double wsum[kMaxWarps][9];
    double *sigp;                       // rank 0's sig
    int item;
    // stall tracker (testing warp): the squared residual that the next ones
    // must reach a quarter of, and the evaluation that set it
    float st_h, st_l;
    long long st_e;
    df thresh2;  // (tol f_ref)^2
};

// Tables of one CTA (shared memory; see mixed_node_smem for the layout).
struct NodeTables {
    float4 *Q;      // increments, two arrays of q_cap
    float4 *G;      // per own free node: (g_ref, 1/m)
    float4 *V;      // (v, a.x)
    float2 *A;      // (a.y, a.z)
    float4 *K0;     // per slot: (r, EA)
    float *K1;      // per slot: q_ref
    float4 *X0;     // the same for slots beyond the shared ones (global memory)
    float *X1;
    uint32_t *PA;   // cluster addresses (array 0) of the copies of own nodes
    uint32_t *PO;   // per own free node: first copy | count << 24
    int *SS;        // per slab + 1: first slot
    uint16_t *NI;   // per slot: index into the increment array
    int ks;         // slots in shared memory
};

// Reciprocal square root and division, with FTZ the forms that flush subnormals to
// zero (fewer instructions): equal where nothing is subnormal (runtime.cu,
// node_range_ok), so RVEs near FP32's limits get the others.
template <bool FTZ>
__device__ __forceinline__ float rsqrt_of(float x) {
    if (!FTZ) return rsqrtf(x);
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
template <bool FTZ>
__device__ __forceinline__ float div_of(float a, float b) {
    if (!FTZ) return __fdividef(a, b);
    float y;
    asm("div.approx.ftz.f32 %0, %1, %2;" : "=f"(y) : "f"(a), "f"(b));
    return y;
}

// Force increments on a node from N row entries, t(d_ref + dd) - t(d_ref) =
// q_ref dd + dq (r + dd), added to g in row order. N independent chains: one is
// about 200 cycles of latency, so one at a time would leave the pipes idle.
// ALT: the order of the fused products in the two inner products that form h. Parts
// beyond the footprint rule (mixed_fp32_smem) have the second one, only so that
// their trajectories keep the bits they have always had.
template <int N, bool ALT, bool FTZ>
__device__ __forceinline__ void entry_forces(float q0, float q1, float q2, const float4 *qj, const float4 *k0,
                                             const float *qref, float &g0, float &g1, float &g2) {
    float t0[N], t1[N], t2[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const float r0 = k0[i].x, r1 = k0[i].y, r2 = k0[i].z, ea = k0[i].w;
        const float lr2 = dot3(r0, r1, r2, r0, r1, r2);
        const float ril = rsqrt_of<FTZ>(lr2);
        const float e0 = fsub(qj[i].x, q0), e1 = fsub(qj[i].y, q1), e2 = fsub(qj[i].z, q2);
        const float h = ALT ? __fmaf_rn(2.f, dot3(r1, r0, r2, e1, e0, e2), dot3(e1, e0, e2, e1, e0, e2))
                            : __fmaf_rn(2.f, dot3(r0, r1, r2, e0, e1, e2), dot3(e0, e1, e2, e0, e1, e2));
        const float l2 = fadd(lr2, h), rl = rsqrt_of<FTZ>(l2);
        const float dq = div_of<FTZ>(fmul(fmul(fmul(ea, h), rl), ril), __fmaf_rn(lr2, ril, fmul(l2, rl)));
        t0[i] = __fmaf_rn(qref[i], e0, fmul(dq, fadd(r0, e0)));
        t1[i] = __fmaf_rn(qref[i], e1, fmul(dq, fadd(r1, e1)));
        t2[i] = __fmaf_rn(qref[i], e2, fmul(dq, fadd(r2, e2)));
    }
#pragma unroll
    for (int i = 0; i < N; ++i) {
        g0 = fadd(g0, t0[i]);
        g1 = fadd(g1, t1[i]);
        g2 = fadd(g2, t2[i]);
    }
}

// The same with the entries' tables in memory; NI, K0, K1 point at the first.
template <int N, bool ALT, bool FTZ>
__device__ __forceinline__ void table_forces(const float4 &qi, const float4 *Qc, const uint16_t *NI, const float4 *K0,
                                             const float *K1, float &g0, float &g1, float &g2) {
    float4 qj[N], k0[N];
    float qref[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        qj[i] = Qc[NI[32 * i]];
        k0[i] = K0[32 * i];
        qref[i] = K1[32 * i];
    }
    entry_forces<N, ALT, FTZ>(qi.x, qi.y, qi.z, qj, k0, qref, g0, g1, g2);
}

// A slab's row sums from memory: w entries per node.
template <int N, bool ALT, bool FTZ>
__device__ __forceinline__ void row_forces(const float4 &qi, const float4 *Qc, const uint16_t *NI, const float4 *K0,
                                           const float *K1, int w, float &g0, float &g1, float &g2) {
    for (; w >= N; w -= N, NI += 32 * N, K0 += 32 * N, K1 += 32 * N)
        table_forces<N, ALT, FTZ>(qi, Qc, NI, K0, K1, g0, g1, g2);
    if (N > 2 && w >= 2) {
        table_forces<2, ALT, FTZ>(qi, Qc, NI, K0, K1, g0, g1, g2);
        w -= 2, NI += 64, K0 += 64, K1 += 64;
    }
    if (w > 0) table_forces<1, ALT, FTZ>(qi, Qc, NI, K0, K1, g0, g1, g2);
}

// One node's state between iterations: half-step velocity, acceleration.
struct Motion {
    float v0, v1, v2, a0, a1, a2;
};

// Acceleration and full-step velocity from the force g (Algorithm 1: damping,
// a = (g + f_d) / m, v += dt/2 a), the residual and kinetic-energy terms, then
// the next partial velocity update; returns the next increment on top of d.
__device__ __forceinline__ float4 node_update(Motion &s, float g0, float g1, float g2, float im, float cf, float hdt,
                                              float dt, float d0, float d1, float d2, bool want_k, float &rs, float &kes) {
    s.a0 = __fmaf_rn(g0, im, -fmul(cf, s.v0));
    s.a1 = __fmaf_rn(g1, im, -fmul(cf, s.v1));
    s.a2 = __fmaf_rn(g2, im, -fmul(cf, s.v2));
    const float w0 = __fmaf_rn(hdt, s.a0, s.v0), w1 = __fmaf_rn(hdt, s.a1, s.v1), w2 = __fmaf_rn(hdt, s.a2, s.v2);
    rs = fadd(rs, dot3(g0, g1, g2, g0, g1, g2));
    if (want_k) kes = fadd(kes, __fdiv_rn(fmul(0.5f, dot3(w0, w1, w2, w0, w1, w2)), im));
    s.v0 = __fmaf_rn(hdt, s.a0, w0);
    s.v1 = __fmaf_rn(hdt, s.a1, w1);
    s.v2 = __fmaf_rn(hdt, s.a2, w2);
    return make_float4(__fmaf_rn(dt, s.v0, d0), __fmaf_rn(dt, s.v1, d1), __fmaf_rn(dt, s.v2, d2), 0.f);
}

// Degrees, slabs, neighbour places and copy lists of this CTA's rows.
__device__ __noinline__ void node_rows(const DevMesh &M, const RveDesc &R, const Part pt, const NodeTables T) {
    const int32_t *rowptr = M.rowptr + R.rp0 + pt.f0;
    const int ns = (pt.nfr + 31) >> 5;
    slab_offsets(T.SS, pt.nfr, [&](int k) { return rowptr[k + 1] - rowptr[k]; });
    const uint32_t q0 = smem_addr(T.Q);
    copy_lists(M, R, pt, T.PO, [&](int x, uint32_t w) { T.PA[x] = cluster_addr(q0 + 16u * (w & 0xffffu), w >> 16); });
    __syncthreads();
    for (int k = threadIdx.x; k < 32 * ns; k += blockDim.x) {
        const int beg = k < pt.nfr ? rowptr[k] : 0, deg = k < pt.nfr ? rowptr[k + 1] - beg : 0;
        int sl = T.SS[k >> 5] + (k & 31);
        const int end = T.SS[(k >> 5) + 1];
        for (int e = 0; sl < end; ++e, sl += 32)
            T.NI[sl] = e < deg ? M.qidx[R.csr0 + beg + e] : (uint16_t)min(k, pt.nfr);
    }
}

// Reference positions x_ref = X + u (FP32 rounding of the double-float sum) of
// this CTA's nodes into the RVE's global scratch; with `fold`, the increments
// of array Qc are added to the double-float displacement first.
__device__ __noinline__ void node_positions(const DevMesh &M, const DevState &S, const RveDesc &R, const Part pt,
                                            const float4 *Qc, bool fold) {
    const int n = R.n_nodes;
    const int64_t b3 = 3 * R.node0;
    float *uh = S.uh + b3, *ul = S.ul + b3, *xr = reinterpret_cast<float *>(S.xg + b3);
    for (int k = threadIdx.x; k < pt.m(); k += blockDim.x) {
        const int i = pt.gidx(k);
        float dd[3] = {0.f, 0.f, 0.f};
        if (fold && k < pt.nfr) {
            const float4 d = Qc[k];
            dd[0] = d.x; dd[1] = d.y; dd[2] = d.z;
        }
        for (int c = 0; c < 3; ++c) {
            df u = {uh[c * n + i], ul[c * n + i]};
            if (fold && k < pt.nfr) {
                u = df_add_f(u, dd[c]);
                uh[c * n + i] = u.hi;
                ul[c * n + i] = u.lo;
            }
            xr[c * n + i] = df_add({M.Xh[b3 + c * n + i], M.Xl[b3 + c * n + i]}, u).hi;
        }
    }
}

// Reference force on own free node i (double-float, displacement form) from
// the displacements in global memory.
__device__ __noinline__ float3 node_gref(const DevMesh &M, const DevState &S, const RveDesc &R, int i) {
    const int n = R.n_nodes;
    const int64_t b3 = 3 * R.node0;
    const float *uh = S.uh + b3, *ul = S.ul + b3;
    const int32_t *rowptr = M.rowptr + R.rp0;
    const df ui0 = {uh[i], ul[i]}, ui1 = {uh[n + i], ul[n + i]}, ui2 = {uh[2 * n + i], ul[2 * n + i]};
    df g0 = df_from(0.f), g1 = df_from(0.f), g2 = df_from(0.f);
    for (int e = rowptr[i]; e < rowptr[i + 1]; ++e) {
        const int64_t kk = R.csr0 + e;
        const int j = M.col[kk];
        df_entry_force(M, kk, df_sub({uh[j], ul[j]}, ui0), df_sub({uh[n + j], ul[n + j]}, ui1),
                       df_sub({uh[2 * n + j], ul[2 * n + j]}, ui2), g0, g1, g2);
    }
    return make_float3(g0.hi, g1.hi, g2.hi);
}

// Row constants of the own free nodes from the reference positions in global
// memory; with `regather` the reference forces too.
template <bool FTZ>
__device__ __noinline__ void node_constants(const DevMesh &M, const DevState &S, const RveDesc &R, const Part pt,
                                            const NodeTables T, bool regather) {
    const int n = R.n_nodes, ns = (pt.nfr + 31) >> 5;
    const int64_t b3 = 3 * R.node0;
    const float *xr = reinterpret_cast<const float *>(S.xg + b3);
    const int32_t *rowptr = M.rowptr + R.rp0 + pt.f0;
    for (int k = threadIdx.x; k < 32 * ns; k += blockDim.x) {
        const int i = pt.f0 + k;
        int beg = 0, deg = 0;
        float x0 = 0.f, x1 = 0.f, x2 = 0.f;
        if (k < pt.nfr) {
            beg = rowptr[k];
            deg = rowptr[k + 1] - beg;
            x0 = xr[i]; x1 = xr[n + i]; x2 = xr[2 * n + i];
            if (regather) {
                const float3 g = node_gref(M, S, R, i);
                T.G[k] = make_float4(g.x, g.y, g.z, T.G[k].w);
            }
        }
        int sl = T.SS[k >> 5] + (k & 31);
        const int end = T.SS[(k >> 5) + 1];
        const bool in = end <= T.ks;
        for (int e = 0; sl < end; ++e, sl += 32) {
            float4 k0 = make_float4(1.f, 0.f, 0.f, 0.f);
            float k1 = 0.f;
            if (e < deg) {
                const int64_t kk = R.csr0 + beg + e;
                const int j = M.col[kk];
                const float2 ei = M.eaf[kk];
                const float r0 = xr[j] - x0, r1 = xr[n + j] - x1, r2 = xr[2 * n + j] - x2;
                const float ril = rsqrt_of<FTZ>(dot3(r0, r1, r2, r0, r1, r2));
                k0 = make_float4(r0, r1, r2, ei.x);
                k1 = fmul(ei.x, fsub(ei.y, ril));
            }
            if (in) {
                T.K0[sl] = k0;
                T.K1[sl] = k1;
            } else {
                T.X0[sl] = k0;
                T.X1[sl] = k1;
            }
        }
    }
}

// End of the solve: outputs, stress (FP64, once per RVE).
struct RingInc {
    const float4 *ring;
    __device__ float4 operator()(int k) const { return ring[k]; }
};
__device__ __noinline__ void node_finish(NodeShared &sh, const DevMesh &M, const DevState &S, const DevResults &O,
                                         const SolveParams &P, int p, const RveDesc &R, const Part pt,
                                         const float4 *ring, int status, int64_t it, df r2, df k2, double f_ref) {
    cg::cluster_group cl = cg::this_cluster();
    double F[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) F[k] = P.F[9 * (int64_t)p + k];
    const RingInc inc = {ring};
    mixed_finish(cl, sh, M, S, O, P, p, R, pt, F, ring != nullptr, inc, status, it, r2, k2, f_ref);
}

}  // namespace

// One RVE. ONE: every warp has at most one slab, whose state and first
// kRegEntries entries per node stay in registers. MINB: CTAs per SM that the
// registers are bounded for. The arithmetic is the same in all of them.
template <bool ONE, int MINB, bool ALT, bool FTZ>
__device__ __forceinline__ void node_rve(NodeShared &sh, const DevMesh &M, const DevState &S, const DevResults &O,
                                         const SolveParams &P, const NodeShape &sp, int p, const NodeTables &T0) {
    cg::cluster_group cl = cg::this_cluster();
    const RveDesc &R = M.rve[p];
    const int C = sp.parts;
    const Part pt = make_part(M, R, p, (int)cl.block_rank(), C);
    const int n = R.n_nodes, nfr = pt.nfr;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
    const bool test_warp = warp == nw - 1;
    const bool want_k = P.want_ke != 0;
    NodeTables T = T0;
    {
        const int64_t x = R.ell0 + (int64_t)pt.me * R.part_slot_max;
        T.X0 = S.ek0 + x;
        T.X1 = S.ek1 + x;
    }
    // increments of the last kRing evaluations (16-byte aligned in the RVE's
    // 72 bytes per node)
    float4 *const ring = reinterpret_cast<float4 *>((reinterpret_cast<uintptr_t>(S.ualt + 9 * R.node0) + 15) &
                                                    ~(uintptr_t)15) + pt.f0;

    int status = O.status[p];
    const int64_t first = O.iters[p];  // evaluation index of the first FP32 iteration
    const double f_ref = O.f_ref[p];
    df r2 = df_from_double(O.rel_res[p]);
    df k2 = df_from_double(O.ke[p]);
    int64_t it = first;
    int fin = -1;  // ring entry of the final state, -1: none
    cl.sync();     // every CTA has read the lead's results before rank 0 rewrites them

    if (status == RVE_PENDING) {
        const double dt64 = dmul(P.alpha, R.dtc);
        const float dt = (float)dt64, hdt = (float)dmul(0.5, dt64), cf = (float)R.c;
        const int K = P.rebase_every > 0 ? P.rebase_every : 512;
        const int nslab = (nfr + 31) >> 5;
        const uint32_t qbytes = 16u * (uint32_t)sp.q_cap;
        node_rows(M, R, pt, T);
        node_positions(M, S, R, pt, nullptr, false);
        {
            const int64_t b3 = 3 * R.node0 + pt.f0;
            const float *vh = S.vh + b3, *ah = S.ah + b3, *fg = S.fg + b3, *imh = M.imh + R.node0 + pt.f0;
            for (int k = threadIdx.x; k < nfr; k += blockDim.x) {
                T.V[k] = make_float4(vh[k], vh[n + k], vh[2 * n + k], ah[k]);
                T.A[k] = make_float2(ah[n + k], ah[2 * n + k]);
                // g_ref = fg from the lead's last force evaluation at exactly this state
                T.G[k] = make_float4(fg[k], fg[n + k], fg[2 * n + k], imh[k]);
            }
        }
        if (threadIdx.x == 0) {
            T.Q[nfr] = T.Q[sp.q_cap + nfr] = make_float4(0.f, 0.f, 0.f, 0.f);
            sh.thresh2 = df_from_double(dmul(dmul(P.tol, f_ref), dmul(P.tol, f_ref)));
            sh.st_h = INFINITY;
            sh.st_l = 0.f;
            sh.st_e = first;
        }
        cl.sync();
        node_constants<FTZ>(M, S, R, pt, T, false);
        // Own node k's increment of the next evaluation (array par) and its
        // copies `po` in other CTAs.
        auto place = [&](int k, const float4 &next, int par, uint32_t po) {
            T.Q[par * sp.q_cap + k] = next;
            const uint32_t off = par ? qbytes : 0u;
            for (uint32_t x = po & 0xffffffu, e = x + (po >> 24); x < e; ++x) st_cluster(T.PA[x] + off, next);
        };
        auto load = [&](int k) {
            const float4 v = T.V[k];
            const float2 a = T.A[k];
            return Motion{v.x, v.y, v.z, v.w, a.x, a.y};
        };
        auto store = [&](int k, const Motion &s) {
            T.V[k] = make_float4(s.v0, s.v1, s.v2, s.a0);
            T.A[k] = make_float2(s.a1, s.a2);
        };
        // the first partial velocity update and displacement
        for (int k = threadIdx.x; k < nfr; k += blockDim.x) {
            Motion s = load(k);
            s.v0 = __fmaf_rn(hdt, s.a0, s.v0);
            s.v1 = __fmaf_rn(hdt, s.a1, s.v1);
            s.v2 = __fmaf_rn(hdt, s.a2, s.v2);
            store(k, s);
            place(k, make_float4(__fmaf_rn(dt, s.v0, 0.f), __fmaf_rn(dt, s.v1, 0.f), __fmaf_rn(dt, s.v2, 0.f), 0.f), 0,
                  T.PO[k]);
        }
        // ONE: the thread's node, its state, row tables and copies
        const int k1 = threadIdx.x, kq = min(k1, nfr);
        const int sl1 = ONE && warp < nslab ? T.SS[warp] + lane : 0;
        const int w1 = ONE && warp < nslab ? (T.SS[warp + 1] - T.SS[warp]) >> 5 : 0;
        Motion mo = {};
        float4 G = {}, q = {}, c0[kRegEntries];
        float c1[kRegEntries];
        int ci[kRegEntries];
        uint32_t po1 = 0;
        auto load_one = [&](int par) {
            if (!ONE) return;
            if (k1 < nfr) {
                mo = load(k1);
                G = T.G[k1];
                po1 = T.PO[k1];
            }
            q = T.Q[par * sp.q_cap + kq];
#pragma unroll
            for (int j = 0; j < kRegEntries; ++j) {
                const bool in = j < w1;
                c0[j] = in ? T.K0[sl1 + 32 * j] : make_float4(1.f, 0.f, 0.f, 0.f);
                c1[j] = in ? T.K1[sl1 + 32 * j] : 0.f;
                ci[j] = in ? T.NI[sl1 + 32 * j] : kq;
            }
        };
        load_one(0);
        int since = 0;        // evaluations since the reference last moved
        int par = 0, sb = 0;  // evaluation ev: array, sums array
        int64_t ev = first;
        for (;; ++ev, ++since, par ^= 1, sb = (sb == 2 ? 0 : sb + 1)) {
            if (C > 1) {
                cluster_arrive();
                cluster_wait();
            } else {
                __syncthreads();
            }
            const bool rebase = since >= K;
            int code = since >= 4 ? sh.vd[par ^ 1].code : -1;  // on evaluation ev - 4
            float4 *const now = ring + (int)(ev & (kRing - 1)) * n;
            float rs = 0.f, kes = 0.f;
            if (code >= 0 || rebase) {
                if (ONE && k1 < nfr) store(k1, mo);
                Verdict v = sh.vd[par ^ 1];
                int back = 4;
                if (code < 0) {
                    // the reference moves: every earlier evaluation is tested
                    // first, by every warp
                    if (test_warp) publish_sums(sh, par ^ 1, sb == 0 ? 2 : sb - 1, pt.me, C, want_k);
                    cl.sync();
                    for (back = min(since, 3); back >= 1; --back) {
                        const int tb = sb - back < 0 ? sb - back + 3 : sb - back;
                        v = sums_verdict(sh, tb, C, sh.thresh2, ev - back + 1, want_k, P.max_iter);
                        code = v.code;
                        if (code >= 0) break;
                    }
                }
                if (code >= 0) {
                    status = code;
                    if (code == RVE_STALLED) {
                        // Hand back at the end of evaluation ev - 1, whose state
                        // is complete: displacement = double-float base + its
                        // increment, acceleration a, full-step velocity = v - dt/2 a.
                        const int64_t b3 = 3 * R.node0 + pt.f0;
                        const float4 *inc = ring + (int)((ev - 1) & (kRing - 1)) * n;
                        for (int k = threadIdx.x; k < nfr; k += blockDim.x) {
                            const Motion s = load(k);
                            const float4 d = inc[k];
                            const float vv[3] = {s.v0, s.v1, s.v2}, aa[3] = {s.a0, s.a1, s.a2}, dd[3] = {d.x, d.y, d.z};
                            for (int c = 0; c < 3; ++c) {
                                const int64_t i = b3 + c * n + k;
                                const df u = df_add_f({S.uh[i], S.ul[i]}, dd[c]);
                                S.uh[i] = u.hi;
                                S.ul[i] = u.lo;
                                S.vh[i] = __fmaf_rn(-hdt, aa[c], vv[c]);
                                S.vl[i] = 0.f;
                                S.ah[i] = aa[c];
                                S.al[i] = 0.f;
                            }
                        }
                        it = ev - 1;
                    } else {
                        fin = (int)((ev - back) & (kRing - 1));
                        it = ev - back + 1;
                        r2 = {v.r2h, v.r2l};
                        k2 = {v.k2h, v.k2l};
                    }
                    break;
                }
                node_positions(M, S, R, pt, T.Q + par * sp.q_cap, true);
                cl.sync();
                node_constants<FTZ>(M, S, R, pt, T, true);
                for (int k = threadIdx.x; k < nfr; k += blockDim.x) {
                    const float4 g = T.G[k];
                    Motion s = load(k);
                    now[k] = make_float4(0.f, 0.f, 0.f, 0.f);
                    const float4 next = node_update(s, g.x, g.y, g.z, g.w, cf, hdt, dt, 0.f, 0.f, 0.f, want_k, rs, kes);
                    store(k, s);
                    place(k, next, par ^ 1, T.PO[k]);
                }
                load_one(par ^ 1);
                since = 0;
            } else {
                const float4 *Qc = T.Q + par * sp.q_cap;
                if (ONE) {
                    if (w1 > 0) {
                        if (k1 < nfr) now[k1] = q;
                        float g0 = 0.f, g1 = 0.f, g2 = 0.f;
                        float4 qj[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) qj[j] = Qc[ci[j]];
                        entry_forces<4, ALT, FTZ>(q.x, q.y, q.z, qj, c0, c1, g0, g1, g2);
                        if (w1 == 5) {
                            qj[0] = Qc[ci[4]];
                            entry_forces<1, ALT, FTZ>(q.x, q.y, q.z, qj, c0 + 4, c1 + 4, g0, g1, g2);
                        } else if (w1 > 5) {
                            qj[0] = Qc[ci[4]];
                            qj[1] = Qc[ci[5]];
                            entry_forces<2, ALT, FTZ>(q.x, q.y, q.z, qj, c0 + 4, c1 + 4, g0, g1, g2);
                            constexpr int x = 32 * kRegEntries;
                            row_forces<4, ALT, FTZ>(q, Qc, T.NI + sl1 + x, T.K0 + sl1 + x, T.K1 + sl1 + x, w1 - kRegEntries, g0, g1, g2);
                        }
                        if (k1 < nfr) {
                            g0 = fadd(g0, G.x); g1 = fadd(g1, G.y); g2 = fadd(g2, G.z);
                            q = node_update(mo, g0, g1, g2, G.w, cf, hdt, dt, q.x, q.y, q.z, want_k, rs, kes);
                            place(k1, q, par ^ 1, po1);
                        }
                    }
                } else {
                    for (int s = warp; s < nslab; s += nw) {
                        const int k = 32 * s + lane;
                        const float4 qi = Qc[min(k, nfr)];
                        const int s0 = T.SS[s], end = T.SS[s + 1], w = (end - s0) >> 5;
                        if (k < nfr) now[k] = qi;
                        float g0 = 0.f, g1 = 0.f, g2 = 0.f;
                        const int sl = s0 + lane;
                        if (MINB > 1 || end <= T.ks) row_forces<MINB == 1 ? 4 : 3, ALT, FTZ>(qi, Qc, T.NI + sl, T.K0 + sl, T.K1 + sl, w, g0, g1, g2);
                        else row_forces<4, ALT, FTZ>(qi, Qc, T.NI + sl, T.X0 + sl, T.X1 + sl, w, g0, g1, g2);
                        if (k < nfr) {
                            const float4 g = T.G[k];
                            Motion m = load(k);
                            g0 = fadd(g0, g.x); g1 = fadd(g1, g.y); g2 = fadd(g2, g.z);
                            const float4 next = node_update(m, g0, g1, g2, g.w, cf, hdt, dt, qi.x, qi.y, qi.z, want_k, rs, kes);
                            store(k, m);
                            place(k, next, par ^ 1, T.PO[k]);
                        }
                    }
                }
                if (test_warp) {
                    // sums of evaluation ev - 1, which every thread left before
                    // this iteration's barrier
                    if (since >= 1) publish_sums(sh, par ^ 1, sb == 0 ? 2 : sb - 1, pt.me, C, want_k);
                    // verdict on evaluation ev - 3, whose sums arrived by this
                    // iteration's barrier or earlier
                    if (since >= 3) {
                        const int64_t chk = ev - 3;
                        Verdict mine = sums_verdict(sh, sb, C, sh.thresh2, chk + 1, want_k, P.max_iter);
                        if (lane == 0) {
                            // Stall check: the squared residual must reach a
                            // quarter of its reference value within
                            // stall_window evaluations, else the RVE goes back
                            // to the double-float kernel (the FP32 increments
                            // have hit their rounding floor). Every CTA's
                            // testing warp sees the same verdicts, so all agree.
                            if (mine.code < 0 && P.stall_window > 0) {
                                const df r2c = {mine.r2h, mine.r2l};
                                if (df_le(r2c, {0.25f * sh.st_h, 0.25f * sh.st_l})) {
                                    sh.st_h = r2c.hi;
                                    sh.st_l = r2c.lo;
                                    sh.st_e = chk;
                                } else if (chk - sh.st_e >= P.stall_window) {
                                    mine.code = RVE_STALLED;
                                }
                            }
                            sh.vd[par] = mine;
                        }
                    }
                }
            }
            sh.rs[par][warp][lane] = rs;
            if (want_k) sh.ke[par][warp][lane] = kes;
        }
    }

    if (status == RVE_STALLED) {
        // handed back to the double-float kernel (resume launch), which
        // finishes the solve and writes every output
        if (pt.me == 0 && threadIdx.x == 0) {
            O.iters[p] = it;
            O.status[p] = RVE_STALLED;
        }
        cl.sync();
        return;
    }
    node_finish(sh, M, S, O, P, p, R, pt, fin >= 0 ? ring + fin * n : nullptr, status, it, r2, k2, f_ref);
}

template <bool ONE, int MINB, bool ALT, bool FTZ>
__global__ void __launch_bounds__(kThreads, MINB)
    dr_mixed_node_kernel(const __grid_constant__ DevMesh M, const __grid_constant__ DevState S,
                         const __grid_constant__ DevResults O, const __grid_constant__ SolveParams P,
                         const __grid_constant__ NodeShape sp) {
    extern __shared__ __align__(16) float4 dsm[];
    __shared__ __align__(16) NodeShared sh;
    cg::cluster_group cl = cg::this_cluster();
    NodeTables T;
    // layout as in mixed_node_smem
    T.Q = dsm;
    T.G = T.Q + 2 * sp.q_cap;
    T.V = T.G + sp.free_cap;
    T.K0 = T.V + sp.free_cap;
    T.A = reinterpret_cast<float2 *>(T.K0 + sp.smem_slots);
    T.K1 = reinterpret_cast<float *>(T.A + sp.free_cap);
    T.PA = reinterpret_cast<uint32_t *>(T.K1 + sp.smem_slots);
    T.PO = T.PA + sp.push_cap;
    T.SS = reinterpret_cast<int *>(T.PO + sp.free_cap);
    T.NI = reinterpret_cast<uint16_t *>(T.SS + sp.free_cap / 32 + 2);
    T.X0 = nullptr;
    T.X1 = nullptr;
    T.ks = sp.smem_slots;
    if (threadIdx.x == 0) sh.sigp = cl.map_shared_rank(&sh.sig[0][0], 0);
    for (;;) {
        if (cl.block_rank() == 0 && threadIdx.x == 0) sh.item = atomicAdd(P.counter + 1, 1);
        cl.sync();
        const int item = *cl.map_shared_rank(&sh.item, 0);
        cl.sync();
        if (item >= P.queue_len) return;
        node_rve<ONE, MINB, ALT, FTZ>(sh, M, S, O, P, sp, P.queue[item], T);
    }
}

namespace {
using NodeKernel = void (*)(DevMesh, DevState, DevResults, SolveParams, NodeShape);

// pair: two CTAs per SM at 64 registers a thread hide each other's barriers and
// gathers, for launches of more clusters than fit at one per SM (runtime.cu).
NodeKernel pick_node(const NodeShape &sp, int block, bool pair) {
    if (!sp.flush) return sp.alt ? dr_mixed_node_kernel<false, 1, true, false> : dr_mixed_node_kernel<false, 1, false, false>;
    if (sp.alt) return dr_mixed_node_kernel<false, 1, true, true>;
    if (pair) return dr_mixed_node_kernel<false, 2, false, true>;
    return sp.free_cap <= block && sp.smem_slots >= sp.slot_cap ? dr_mixed_node_kernel<true, 1, false, true>
                                                                : dr_mixed_node_kernel<false, 1, false, true>;
}

cudaLaunchConfig_t node_config(int clusters, int parts, int block, size_t smem, cudaLaunchAttribute *attr,
                               cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(clusters * parts, 1, 1);
    cfg.blockDim = dim3(block, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = parts;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

// Raise a kernel's dynamic shared-memory limit (and allow 16-CTA clusters)
// once per device and size, so that launches recorded into a CUDA graph make
// no attribute calls of their own.
std::mutex g_node_mutex;
std::map<std::pair<const void *, int>, int> g_node_bytes;

void prepare_node(NodeKernel k, size_t smem) {
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lock(g_node_mutex);
    int &have = g_node_bytes[{reinterpret_cast<const void *>(k), dev}];
    if (have == 0 || have < (int)smem) {
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        have = std::max(have, (int)smem);
    }
}
}  // namespace

size_t mixed_node_smem(const NodeShape &sp) {
    const size_t q = (size_t)sp.q_cap, F = (size_t)sp.free_cap;
    const size_t b = 16 * (2 * q + 2 * F + (size_t)sp.smem_slots) + 8 * F + 4 * (size_t)sp.smem_slots +
                     4 * (size_t)sp.push_cap + 4 * F + 4 * (F / 32 + 2) + 2 * (size_t)sp.slot_cap;
    return (b + 15) & ~size_t(15);
}

int launch_dr_mixed_node(const DevMesh &m, const DevState &s, const DevResults &r, const SolveParams &p,
                         int clusters, int block, size_t smem, const NodeShape &sp, bool pair, void *stream) {
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = node_config(clusters, sp.parts, block, smem, attr, static_cast<cudaStream_t>(stream));
    const NodeKernel k = pick_node(sp, block, pair);
    prepare_node(k, smem);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k, m, s, r, p, sp);
    if (e != cudaSuccess) return (int)e;
    return (int)cudaGetLastError();
}

int occupancy_dr_mixed_node(int block, size_t smem, const NodeShape &sp, bool pair) {
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = node_config(64, sp.parts, block, smem, attr, nullptr);
    const NodeKernel k = pick_node(sp, block, pair);
    prepare_node(k, smem);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

}  // namespace fe2
