// Mixed-precision dynamic relaxation (Algorithm 1) for a batch of RVEs: one
// thread-block cluster per RVE, three persistent launches per size class (the
// double-float lead, the FP32 phase, the double-float resume of stalled RVEs).
//
// The lead runs in dr_mixed_lead.cu's kernel and the FP32 phase in
// dr_mixed_node.cu's, both with their tables on chip. The kernels of this file,
// which re-read the CSR rows from L2, remain for parts whose displacements or
// increments (with the copies of neighbours in other parts) do not fit in shared
// memory.
//
// Layout. The RVE is split spatially into `parts` pieces, one per CTA of the
// cluster; a CTA stages the state of its own nodes in its shared memory and (in
// this file) reads neighbours owned by other CTAs through distributed shared
// memory. The
// paper used one thread team per sub-problem (Section III); a cluster lets one
// sub-problem span several SMs.
//
// Precision. All arithmetic of the iterations runs on the FP32 pipes (GB300
// issues FP64 at roughly 1/70 of the FP32 rate):
//  * lead kernel: double-float (hi + lo FP32 pairs, ~48 bits) displacement,
//    velocity, acceleration and element forces until the relative residual
//    first drops below lead_tol. Random fiber networks are not isostatic and
//    can pass bifurcation points (Section II); which equilibrium the
//    relaxation settles into is decided in this transient and is sensitive to
//    force errors far below FP32 rounding. Element forces are evaluated in
//    displacement form, d = D + (u_j - u_i) with D = X_j - X_i, and
//    N/l = EA h / (L l (l + L)), h = l^2 - L^2 = (u_j - u_i).(D + d), which
//    has no cancellation, so the double-float strain is accurate to ~1e-14;
//  * FP32 kernel: each element force is an exact increment about a reference
//    state x_ref,
//        t(d_ref + dd) = t(d_ref) + q_ref dd + dq (d_ref + dd),
//        q = N/l = EA (1/L - 1/l),  dq = EA h / (l l_ref (l + l_ref)),
//        h = l^2 - l_ref^2 = 2 d_ref.dd + dd.dd,
//    so every FP32 operation acts on small quantities; the nodal sums of
//    t(d_ref) (g_ref) are evaluated in double-float every rebase_every
//    iterations, when the FP32 increment du is folded into the double-float
//    displacement. Velocity and increment updates are FP32;
//  * the residual norm is summed per warp in FP32 (squares, no cancellation)
//    and across warps and CTAs in double-float; the threshold (tol f_ref)^2 is
//    formed in FP64 once per RVE; the stress sum is FP64.
//
// Synchronisation of this file's FP32 kernel. One cluster barrier per
// iteration. Five displacement-increment buffers rotate. Each node's owner
// thread computes the next iteration's increment right after the node's
// velocity update, so an iteration begins at the barrier. Between the
// barrier's arrive and wait, every warp publishes its residual partial of the
// previous evaluation to its own CTA, and one warp per CTA totals evaluation
// n-3 across the cluster (DSMEM reads) and leaves a verdict. All warps read
// the verdict after the next barrier. If the test succeeded, they finish with
// the state of the tested evaluation, whose buffer is still intact.
#include <cooperative_groups.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <utility>

#include "dr_mixed.cuh"

namespace fe2 {

namespace {

constexpr int kLeadBufs = 3;   // lead kernel: rotating partial buffers
// FP32 kernel without row tables (this file): shared memory per node, the
// reference position and five increment buffers (float4 each); velocity and
// acceleration live in global memory.
constexpr size_t kFp32PlainNodeBytes = (1 + kBufs) * sizeof(float4);
// Per-node bytes of the footprint rule that sets the cluster size
// (mixed_fp32_smem).
constexpr size_t kFp32NodeBytes = (1 + kBufs + 1) * sizeof(float4) + sizeof(float2);
// Lead kernel without tables (this file): shared memory per node, one
// double-float displacement (hi, lo float4).
constexpr size_t kLeadPlainNodeBytes = 2 * sizeof(float4);
__host__ __device__ constexpr size_t align16(size_t x) { return (x + 15) & ~size_t(15); }

struct MixedShared {
    // lead kernel: per-warp residual partials of every CTA, dense: entry
    // (rank * warps + warp)
    float red[kLeadBufs][kMaxParts * kMaxWarps];
    float kred[kLeadBufs][kMaxParts * kMaxWarps]; // kinetic-energy partials
    // FP32 kernel: this CTA's per-warp partials (residual, kinetic energy)
    float own[kBufs][2][kMaxWarps];
    Verdict vd[kBufs];                        // verdicts of the testing warp
    float *ownp[kMaxParts];                   // every CTA's own
    double sig[kMaxParts][9];                 // stress partials, read by rank 0
    double wsum[kMaxWarps][9];                // per-warp stress partials
    float4 *P[kMaxParts];                     // every CTA's position array
    float4 *Q[kBufs][kMaxParts];              // every CTA's increment / low-part arrays
    float *redp[kMaxParts];                   // every CTA's red
    float *kredp[kMaxParts];                  // every CTA's kred
    double *sigp;                             // rank 0's sig
    int item;
    // FP32 kernel stall tracker (testing warp): the squared residual that the
    // next ones must reach a quarter of, and the evaluation that set it
    float st_h, st_l;
    long long st_e;
};

// Double-float total of the cluster's per-warp partials (buffer `buf`),
// computed warp-parallel on the FP32 pipes: lane l adds entries l, l+32, ...
// and a butterfly of double-float additions finishes the sum. The order is
// fixed, so every warp of every CTA obtains the same bits. GB300 issues FP64
// at a small fraction of its FP32 rate, which would make an FP64 reduction by
// every thread cost more than the iteration itself.
__device__ __forceinline__ df cluster_total(const float (*red)[kMaxParts * kMaxWarps], int buf, int C) {
    const int total = C * (int)(blockDim.x >> 5);
    const int lane = threadIdx.x & 31;
    df acc = df_from(0.f);
    for (int j = lane; j < total; j += 32) acc = df_add_f(acc, red[buf][j]);
    for (int o = 16; o > 0; o >>= 1) {
        const df other = {__shfl_xor_sync(0xffffffffu, acc.hi, o), __shfl_xor_sync(0xffffffffu, acc.lo, o)};
        acc = df_add(acc, other);
    }
    return acc;
}

// Publish this thread's FP32 partials (warp-reduced) into every CTA's buffer.
__device__ __forceinline__ void publish(MixedShared &sh, const Part &pt, float v, float kv, bool want_k,
                                        int buf) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (want_k)
        for (int o = 16; o > 0; o >>= 1) kv += __shfl_xor_sync(0xffffffffu, kv, o);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int slot = buf * (kMaxParts * kMaxWarps) + pt.me * (int)(blockDim.x >> 5) + warp;
    if (lane < pt.C) {
        sh.redp[lane][slot] = v;
        if (want_k) sh.kredp[lane][slot] = kv;
    }
}

// Combine double-float partial sums over groups of L consecutive lanes (every
// lane of the warp must call this).
__device__ __forceinline__ void df_group_sum(df &g0, df &g1, df &g2, int L) {
    for (int o = 1; o < L; o <<= 1) {
        const df a0 = {__shfl_xor_sync(0xffffffffu, g0.hi, o), __shfl_xor_sync(0xffffffffu, g0.lo, o)};
        const df a1 = {__shfl_xor_sync(0xffffffffu, g1.hi, o), __shfl_xor_sync(0xffffffffu, g1.lo, o)};
        const df a2 = {__shfl_xor_sync(0xffffffffu, g2.hi, o), __shfl_xor_sync(0xffffffffu, g2.lo, o)};
        g0 = df_add(g0, a0);
        g1 = df_add(g1, a1);
        g2 = df_add(g2, a2);
    }
}

// Double-float internal force on own node k (Algorithm 1, getInternalForces)
// in displacement form; the node's and its neighbours' displacements are
// staged as (hi, lo) in (Pl, Ql) and the other CTAs' copies (Q buffer qbuf).
__device__ __forceinline__ void gather_df(const DevMesh &M, const RveDesc &R, const int32_t *rowptr,
                                          const MixedShared &sh, const Part &pt, int k,
                                          const float4 *Pl, const float4 *Ql, int qbuf, df &g0,
                                          df &g1, df &g2, int sub = 0, int L = 1) {
    const int gi = pt.gidx(k);
    const float4 pi = Pl[k], qi = Ql[k];
    const df ui0 = {pi.x, qi.x}, ui1 = {pi.y, qi.y}, ui2 = {pi.z, qi.z};
    g0 = df_from(0.f); g1 = df_from(0.f); g2 = df_from(0.f);
    const int beg = rowptr[gi], end = rowptr[gi + 1];
    // lane `sub` of L takes edges sub, sub+L, ... (the caller combines the lanes)
    for (int e = beg + sub; e < end; e += L) {
        const int64_t kk = R.csr0 + e;
        const int cp = M.col_part[kk];
        const int r = cp >> 16, loc = cp & 0xffff;
        const float4 pj = r == pt.me ? Pl[loc] : sh.P[r][loc];
        const float4 qj = r == pt.me ? Ql[loc] : sh.Q[qbuf][r][loc];
        df_entry_force(M, kk, df_sub({pj.x, qj.x}, ui0), df_sub({pj.y, qj.y}, ui1), df_sub({pj.z, qj.z}, ui2),
                       g0, g1, g2);
    }
}

__device__ __forceinline__ void map_remote(cg::cluster_group &cl, MixedShared &sh, float4 *Pl,
                                           float4 *const *Qb, int C) {
    if ((int)threadIdx.x < C) {
        const int r = threadIdx.x;
        sh.P[r] = cl.map_shared_rank(Pl, r);
        for (int b = 0; b < kBufs; ++b) sh.Q[b][r] = cl.map_shared_rank(Qb[b], r);
        sh.redp[r] = cl.map_shared_rank(&sh.red[0][0], r);
        sh.kredp[r] = cl.map_shared_rank(&sh.kred[0][0], r);
        sh.ownp[r] = cl.map_shared_rank(&sh.own[0][0][0], r);
    }
    if (threadIdx.x == 0) sh.sigp = cl.map_shared_rank(&sh.sig[0][0], 0);
}

// Next work item of the cluster (rank 0 pops, everyone reads it).
__device__ __forceinline__ int next_item(cg::cluster_group &cl, MixedShared &sh, int32_t *counter) {
    if (cl.block_rank() == 0 && threadIdx.x == 0) sh.item = atomicAdd(counter, 1);
    cl.sync();
    const int item = *cl.map_shared_rank(&sh.item, 0);
    cl.sync();
    return item;
}

// FP32 increment of one element's force on node i from neighbour j about the
// reference state: t(d_ref + dd) - t(d_ref) + q_ref dd, accumulated into g.
// p* hold FP32 reference positions, q* the FP32 displacement increments;
// ei = (EA, 1/L).
__device__ __forceinline__ void edge_increment(const float4 &pi, const float4 &qi, const float4 &pj,
                                               const float4 &qj, float2 ei, float &g0, float &g1,
                                               float &g2) {
    const float r0 = pj.x - pi.x, r1 = pj.y - pi.y, r2 = pj.z - pi.z;
    const float e0 = qj.x - qi.x, e1 = qj.y - qi.y, e2 = qj.z - qi.z;
    const float lr2 = r0 * r0 + r1 * r1 + r2 * r2;
    const float ril = rsqrtf(lr2);
    const float lr = lr2 * ril;
    const float qref = ei.x * (ei.y - ril);
    const float h = 2.f * (r0 * e0 + r1 * e1 + r2 * e2) + (e0 * e0 + e1 * e1 + e2 * e2);
    const float rl = rsqrtf(lr2 + h);
    const float l = (lr2 + h) * rl;
    const float dq = __fdividef(ei.x * h * rl * ril, l + lr);
    g0 += qref * e0 + dq * (r0 + e0);
    g1 += qref * e1 + dq * (r1 + e1);
    g2 += qref * e2 + dq * (r2 + e2);
}

// No FP32 increment on top of the double-float displacement.
struct NoInc {
    __device__ float4 operator()(int) const { return make_float4(0.f, 0.f, 0.f, 0.f); }
};

// ---------------------------------------------------------------------------
// lead kernel: setup (Algorithm 1 lines up to the loop) and the double-float
// iterations
// ---------------------------------------------------------------------------
__device__ void lead_rve(cg::cluster_group &cl, MixedShared &sh, const DevMesh &M, const DevState &S,
                         const DevResults &O, const SolveParams &P, int p, float4 *Pl, float4 *Q0,
                         int &rb) {
    const RveDesc R = M.rve[p];
    const Part pt = make_part(M, R, p, (int)cl.block_rank(), (int)cl.num_blocks());
    const int n = R.n_nodes, m = pt.m();
    const int64_t n0 = R.node0, b3 = 3 * n0;
    const int32_t *rowptr = M.rowptr + R.rp0;
    double F[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) F[k] = P.F[9 * (int64_t)p + k];
    float *uh = S.uh + b3, *ul = S.ul + b3, *vh = S.vh + b3, *vl = S.vl + b3;
    float *ah = S.ah + b3, *al = S.al + b3, *fg = S.fg + b3;
    const float *imh = M.imh + n0, *iml = M.iml + n0;
    const bool want_k = P.want_ke != 0;
    double f_ref = 0.0;
    int64_t it = 0;
    if (P.resume) {
        // resume launch: only RVEs the FP32 phase handed back, from the state
        // it left (double-float displacement, velocity, acceleration)
        const int st0 = O.status[p];
        f_ref = O.f_ref[p];
        it = O.iters[p];
        cl.sync();  // every CTA has read the status before rank 0 rewrites it
        if (st0 != RVE_STALLED) return;
        for (int k = threadIdx.x; k < m; k += blockDim.x) {
            const int i = pt.gidx(k);
            Pl[k] = make_float4(uh[i], uh[n + i], uh[2 * n + i], 0.f);
            Q0[k] = make_float4(ul[i], ul[n + i], ul[2 * n + i], 0.f);
        }
        cl.sync();
    } else {
    // affine displacement (F - I) X for f_ref, and the initial displacement
    for (int k = threadIdx.x; k < m; k += blockDim.x) {
        const int i = pt.gidx(k);
        const double X[3] = {M.X0[n0 + i], M.X1[n0 + i], M.X2[n0 + i]};
        const double *uw[3] = {S.u0 + n0, S.u1 + n0, S.u2 + n0};
        df ua[3];
        const bool fixed = k >= pt.nfr;
        for (int r = 0; r < 3; ++r) {
            const double xa = dadd(dadd(dmul(F[3 * r], X[0]), dmul(F[3 * r + 1], X[1])), dmul(F[3 * r + 2], X[2]));
            const double uaff = dsub(xa, X[r]);
            ua[r] = df_from_double(uaff);
            double u;
            if (fixed || P.init == 1) u = uaff;
            else if (P.init == 2) u = uw[r][i];
            else u = 0.0;
            const df ud = df_from_double(u);
            uh[r * n + i] = ud.hi;
            ul[r * n + i] = ud.lo;
        }
        Pl[k] = make_float4(ua[0].hi, ua[1].hi, ua[2].hi, 0.f);
        Q0[k] = make_float4(ua[0].lo, ua[1].lo, ua[2].lo, 0.f);
    }
    cl.sync();
    float acc = 0.f;
    for (int k = threadIdx.x; k < m; k += blockDim.x) {
        df g0, g1, g2;
        gather_df(M, R, rowptr, sh, pt, k, Pl, Q0, 0, g0, g1, g2);
        acc += g0.hi * g0.hi + g1.hi * g1.hi + g2.hi * g2.hi;
    }
    publish(sh, pt, acc, 0.f, false, rb);
    cl.sync();
    const double f_aff = sqrt(df_to_double(cluster_total(sh.red, rb, pt.C)));
    rb = (rb + 1) % kLeadBufs;
    for (int k = threadIdx.x; k < m; k += blockDim.x) {
        const int i = pt.gidx(k);
        Pl[k] = make_float4(uh[i], uh[n + i], uh[2 * n + i], 0.f);
        Q0[k] = make_float4(ul[i], ul[n + i], ul[2 * n + i], 0.f);
    }
    cl.sync();
    acc = 0.f;
    for (int k = threadIdx.x; k < m; k += blockDim.x) {
        df g[3];
        gather_df(M, R, rowptr, sh, pt, k, Pl, Q0, 0, g[0], g[1], g[2]);
        acc += g[0].hi * g[0].hi + g[1].hi * g[1].hi + g[2].hi * g[2].hi;
        if (k < pt.nfr) {
            const int i = pt.gidx(k);
            const df im = {imh[i], iml[i]};
            for (int r = 0; r < 3; ++r) {
                const df a = df_mul(g[r], im);
                ah[r * n + i] = a.hi; al[r * n + i] = a.lo;
                vh[r * n + i] = 0.f; vl[r * n + i] = 0.f;
                fg[r * n + i] = g[r].hi;
            }
        }
    }
    publish(sh, pt, acc, 0.f, false, rb);
    cl.sync();
    const double f0 = sqrt(df_to_double(cluster_total(sh.red, rb, pt.C)));
    rb = (rb + 1) % kLeadBufs;
    f_ref = f_aff > f0 ? f_aff : f0;
    }
    const df thresh2 = df_from_double(dmul(dmul(P.tol, f_ref), dmul(P.tol, f_ref)));
    // a resumed RVE runs in double-float until it converges
    const df lead2 = P.resume ? thresh2 : df_from_double(dmul(dmul(P.lead_tol, f_ref), dmul(P.lead_tol, f_ref)));
    const int64_t lead_iters = P.resume ? -1 : P.lead_iters;
    const double dt64 = dmul(P.alpha, R.dtc);
    const df dt = df_from_double(dt64), hdt = df_from_double(dmul(0.5, dt64));
    const df cdf = df_from_double(R.c);

    const int64_t it0 = it;
    int status = RVE_PENDING;
    df r2 = df_from(0.f), k2 = df_from(0.f);
    // L lanes share a node's edges; lane 0 of group k owns node k's state in
    // every phase, so consecutive phases need no barrier between them.
    int L = 1;
    while (L < 4 && (int)blockDim.x >= 2 * L * R.part_free_max) L *= 2;
    const int sub = threadIdx.x & (L - 1), grp = threadIdx.x / L, ngrp = blockDim.x / L;
    for (;;) {
        for (int k = grp; k < pt.nfr; k += ngrp) {
            if (sub != 0) continue;
            const int i = pt.f0 + k;
            df u[3];
            for (int c = 0; c < 3; ++c) {
                df v = {vh[c * n + i], vl[c * n + i]};
                const df a = {ah[c * n + i], al[c * n + i]};
                v = df_add(v, df_mul(hdt, a));
                u[c] = df_add({uh[c * n + i], ul[c * n + i]}, df_mul(dt, v));
                vh[c * n + i] = v.hi; vl[c * n + i] = v.lo;
                uh[c * n + i] = u[c].hi; ul[c * n + i] = u[c].lo;
            }
            Pl[k] = make_float4(u[0].hi, u[1].hi, u[2].hi, 0.f);
            Q0[k] = make_float4(u[0].lo, u[1].lo, u[2].lo, 0.f);
        }
        cl.sync();
        float rs = 0.f, kes = 0.f;
        for (int kb = 0; kb < pt.nfr; kb += ngrp) {
            const int k = kb + grp;
            const bool valid = k < pt.nfr;
            df g[3] = {df_from(0.f), df_from(0.f), df_from(0.f)};
            if (valid) gather_df(M, R, rowptr, sh, pt, k, Pl, Q0, 0, g[0], g[1], g[2], sub, L);
            df_group_sum(g[0], g[1], g[2], L);
            if (!valid || sub != 0) continue;
            const int i = pt.f0 + k;
            const df im = {imh[i], iml[i]};
            float vv = 0.f;
            for (int c = 0; c < 3; ++c) {
                df v = {vh[c * n + i], vl[c * n + i]};
                const df a = df_sub(df_mul(g[c], im), df_mul(cdf, v));
                v = df_add(v, df_mul(hdt, a));
                ah[c * n + i] = a.hi; al[c * n + i] = a.lo;
                vh[c * n + i] = v.hi; vl[c * n + i] = v.lo;
                fg[c * n + i] = g[c].hi;
                rs += g[c].hi * g[c].hi;
                vv += v.hi * v.hi;
            }
            if (want_k) kes += 0.5f * vv / imh[i];
        }
        publish(sh, pt, rs, kes, want_k, rb);
        cl.sync();
        r2 = cluster_total(sh.red, rb, pt.C);
        if (want_k) k2 = cluster_total(sh.kred, rb, pt.C);
        rb = (rb + 1) % kLeadBufs;
        ++it;
        if (!isfinite(r2.hi)) { status = RVE_NAN; break; }
        if (df_le(r2, thresh2)) { status = RVE_OK; break; }
        if (it >= P.max_iter) { status = RVE_MAXITER; break; }
        if (lead_iters >= 0 ? it >= lead_iters : df_le(r2, lead2)) break;
    }
    if (P.resume) {
        if (pt.me == 0 && threadIdx.x == 0) O.lead[p] += it - it0;
        mixed_finish(cl, sh, M, S, O, P, p, R, pt, F, false, NoInc{}, status, it, r2, k2, f_ref);
        return;
    }
    if (pt.me == 0 && threadIdx.x == 0) {
        O.iters[p] = it;
        O.lead[p] = it;
        O.status[p] = status;
        O.f_ref[p] = f_ref;
        O.rel_res[p] = df_to_double(r2);  // squared residual, finished by the FP32 kernel
        O.ke[p] = want_k ? df_to_double(k2) : 0.0;
    }
    cl.sync();
}

// ---------------------------------------------------------------------------
// FP32 kernel: increment iterations, reference refreshes, final state, stress
// ---------------------------------------------------------------------------
__device__ void fp32_rve(cg::cluster_group &cl, MixedShared &sh, const DevMesh &M, const DevState &S,
                         const DevResults &O, const SolveParams &P, int p, float4 *Pl,
                         float4 *const *Qb) {
    const RveDesc R = M.rve[p];
    const Part pt = make_part(M, R, p, (int)cl.block_rank(), (int)cl.num_blocks());
    const int n = R.n_nodes, m = pt.m();
    const int64_t n0 = R.node0, b3 = 3 * n0;
    const int32_t *rowptr = M.rowptr + R.rp0;
    // velocity (+ a.x) and a.yz of the own free nodes: global (L2-resident)
    // arrays, which keeps the shared memory at 96 bytes per node
    float4 *SV = S.sv + n0 + pt.f0;
    float2 *SA = S.sa + n0 + pt.f0;
    const float *Xh = M.Xh + b3, *Xl = M.Xl + b3;
    float *uh = S.uh + b3, *ul = S.ul + b3, *vh = S.vh + b3, *ah = S.ah + b3, *fg = S.fg + b3;
    const float *imh = M.imh + n0;
    const bool want_k = P.want_ke != 0;
    double F[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) F[k] = P.F[9 * (int64_t)p + k];

    int status = O.status[p];
    int64_t it = O.iters[p];
    const double f_ref = O.f_ref[p];
    df r2 = df_from_double(O.rel_res[p]);
    df k2 = df_from_double(O.ke[p]);
    int fin = -1;  // increment buffer holding the final state, -1: none
    cl.sync();     // every CTA has read the lead's results before rank 0 rewrites them

    if (status == RVE_PENDING) {
        const df thresh2 = df_from_double(dmul(dmul(P.tol, f_ref), dmul(P.tol, f_ref)));
        const double dt64 = dmul(P.alpha, R.dtc);
        const float dtf = (float)dt64, hdtf = (float)dmul(0.5, dt64), cf = (float)R.c;
        const int K = P.rebase_every > 0 ? P.rebase_every : 512;
        // lanes per node: as many as the CTA size allows for this RVE's largest
        // part. Node k's velocity and
        // acceleration are owned by lane 0 of group k in every phase, so
        // consecutive phases need no barrier between them.
        int lanes = 1;
        while (lanes < 4 && (int)blockDim.x >= 2 * lanes * R.part_free_max) lanes *= 2;
        const int L = lanes;
        const int sub = threadIdx.x & (L - 1), grp = threadIdx.x / L, ngrp = blockDim.x / L;
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        const bool test_warp = warp == (int)(blockDim.x >> 5) - 1;
        // x_ref = X + u (FP32 rounding of the double-float sum), increments zero;
        // g_ref = fg from the lead's last force evaluation at exactly this state
        for (int k = threadIdx.x; k < m; k += blockDim.x) {
            const int i = pt.gidx(k);
            float xr[3];
            for (int c = 0; c < 3; ++c)
                xr[c] = df_add({Xh[c * n + i], Xl[c * n + i]}, {uh[c * n + i], ul[c * n + i]}).hi;
            Pl[k] = make_float4(xr[0], xr[1], xr[2], 0.f);
            for (int b = 0; b < kBufs; ++b) Qb[b][k] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (k < pt.nfr) {
                SV[k] = make_float4(vh[i], vh[n + i], vh[2 * n + i], ah[i]);
                SA[k] = make_float2(ah[n + i], ah[2 * n + i]);
            }
        }
        if (threadIdx.x == 0) {
            sh.st_h = INFINITY;
            sh.st_l = 0.f;
            sh.st_e = it;
        }
        cl.sync();
        const int64_t first = it;  // evaluation index of the first FP32 iteration
        int64_t chk = first;       // next evaluation whose residual is still untested
        int chkb = 0;              // its buffer
        // the verdict the testing warp wrote in the previous iteration
        bool vpend = false;
        int64_t veval = 0;
        int vbuf = 0;
        int since = 0;
        const int32_t *colp = M.col_part + R.csr0;
        const float2 *eafp = M.eaf + R.csr0;
        // Partial velocity update and displacement increment of the first
        // iteration; every later one is done by the node's owner right after
        // the node's velocity update of the previous iteration (the values are
        // still in registers), so an iteration begins at the barrier.
        for (int k = grp; k < pt.nfr; k += ngrp) {
            if (sub != 0) continue;
            const float4 va = SV[k];
            const float2 a12 = SA[k];
            next_increment(va.x, va.y, va.z, va.w, a12.x, a12.y, make_float4(0.f, 0.f, 0.f, 0.f),
                           hdtf, dtf, SV[k], SA[k], Qb[0][k]);
        }
        int b = 0;  // buffer of evaluation nidx
        float part_rs = 0.f, part_ke = 0.f;  // this thread's partials of evaluation nidx-1
        int part_b = -1;                     // and their buffer (-1: none yet)
        for (int64_t nidx = first; status == RVE_PENDING; ++nidx, b = (b + 1 == kBufs ? 0 : b + 1)) {
            const int bn = b + 1 == kBufs ? 0 : b + 1;  // buffer of evaluation nidx + 1
            const int bp = b == 0 ? kBufs - 1 : b - 1;  // buffer of evaluation nidx - 1
            const bool rebase = since >= K;
            cluster_arrive();
            // While the barrier completes: the per-warp residual partials of
            // evaluation nidx-1 go to this CTA's buffer, and evaluation nidx-3
            // (whose partials every CTA has published one barrier ago) is
            // tested by one warp per CTA, whose verdict the others read after
            // the next barrier; before a rebase by every warp. Buffers rotate
            // through five, so the state of a tested evaluation is intact
            // until its verdict is read.
            if (part_b >= 0) {
                for (int o = 16; o > 0; o >>= 1) part_rs += __shfl_xor_sync(0xffffffffu, part_rs, o);
                if (want_k)
                    for (int o = 16; o > 0; o >>= 1) part_ke += __shfl_xor_sync(0xffffffffu, part_ke, o);
                if (lane == 0) {
                    sh.own[part_b][0][warp] = part_rs;
                    if (want_k) sh.own[part_b][1][warp] = part_ke;
                }
            }
            bool tnow = false;
            int64_t teval = 0;
            int tbuf = 0;
            Verdict mine = {-1, 0.f, 0.f, 0.f, 0.f};
            if (chk <= nidx - 3) {
                if (rebase || test_warp) mine = residual_verdict(sh, pt, chkb, chk + 1, thresh2, want_k, P.max_iter);
                if (!rebase && test_warp && lane == 0) {
                    // Stall check: the squared residual must reach a quarter of
                    // its reference value within stall_window evaluations,
                    // else the RVE goes back to the double-float kernel (the
                    // FP32 increments have hit their rounding floor). Every
                    // CTA's testing warp sees the same verdicts, so all agree.
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
                    sh.vd[b] = mine;
                }
                tnow = true; teval = chk; tbuf = chkb;
                ++chk;
                chkb = chkb + 1 == kBufs ? 0 : chkb + 1;
            }
            cluster_wait();
            Verdict stopv = {-1, 0.f, 0.f, 0.f, 0.f};
            int64_t seval = 0;
            int sbuf = 0;
            if (vpend) {
                const Verdict v = sh.vd[bp];
                if (v.code >= 0) { stopv = v; seval = veval; sbuf = vbuf; }
            }
            vpend = false;
            if (stopv.code < 0 && rebase) {
                // the reference moves: every earlier evaluation is tested first
                if (tnow && mine.code >= 0) { stopv = mine; seval = teval; sbuf = tbuf; }
                if (stopv.code < 0 && chk == nidx - 2) {  // published one barrier ago
                    mine = residual_verdict(sh, pt, chkb, chk + 1, thresh2, want_k, P.max_iter);
                    if (mine.code >= 0) { stopv = mine; seval = chk; sbuf = chkb; }
                    ++chk;
                    chkb = chkb + 1 == kBufs ? 0 : chkb + 1;
                }
                if (stopv.code < 0 && chk == nidx - 1) {  // published in this barrier's window
                    cl.sync();
                    mine = residual_verdict(sh, pt, chkb, chk + 1, thresh2, want_k, P.max_iter);
                    if (mine.code >= 0) { stopv = mine; seval = chk; sbuf = chkb; }
                    ++chk;
                    chkb = chkb + 1 == kBufs ? 0 : chkb + 1;
                }
            }
            if (stopv.code == RVE_STALLED) {
                // Hand back at the end of evaluation nidx-1, whose state is
                // complete: displacement = double-float base + its increment
                // (buffer bp), acceleration a, full-step velocity = SV - dt/2 a.
                const float4 *inc = Qb[bp];
                for (int k = grp; k < pt.nfr; k += ngrp) {
                    if (sub != 0) continue;
                    const int i = pt.f0 + k;
                    const float4 d = inc[k], va = SV[k];
                    const float2 ay = SA[k];
                    const float dd[3] = {d.x, d.y, d.z}, vv[3] = {va.x, va.y, va.z}, aa[3] = {va.w, ay.x, ay.y};
                    for (int c = 0; c < 3; ++c) {
                        const df u = df_add_f({uh[c * n + i], ul[c * n + i]}, dd[c]);
                        uh[c * n + i] = u.hi;
                        ul[c * n + i] = u.lo;
                        S.vh[b3 + c * n + i] = vv[c] - hdtf * aa[c];
                        S.vl[b3 + c * n + i] = 0.f;
                        S.ah[b3 + c * n + i] = aa[c];
                        S.al[b3 + c * n + i] = 0.f;
                    }
                }
                status = RVE_STALLED;
                it = nidx - 1;
                break;
            }
            if (stopv.code >= 0) {
                status = stopv.code;
                fin = sbuf;
                it = seval + 1;
                r2 = {stopv.r2h, stopv.r2l};
                k2 = {stopv.k2h, stopv.k2l};
                break;
            }
            float4 *cur = Qb[b];
            float rs = 0.f, kes = 0.f;
            if (rebase) {
                // fold the increment into the double-float displacement; stage
                // double-float displacements (hi in Pl, lo in buffer b)
                for (int k = threadIdx.x; k < m; k += blockDim.x) {
                    const int i = pt.gidx(k);
                    const float4 d = cur[k];
                    const float dd[3] = {d.x, d.y, d.z};
                    df u[3];
                    for (int c = 0; c < 3; ++c) {
                        u[c] = {uh[c * n + i], ul[c * n + i]};
                        if (k < pt.nfr) {
                            u[c] = df_add_f(u[c], dd[c]);
                            uh[c * n + i] = u[c].hi; ul[c * n + i] = u[c].lo;
                        }
                    }
                    Pl[k] = make_float4(u[0].hi, u[1].hi, u[2].hi, 0.f);
                    cur[k] = make_float4(u[0].lo, u[1].lo, u[2].lo, 0.f);
                }
                cl.sync();
                for (int k = threadIdx.x; k < pt.nfr; k += blockDim.x) {
                    const int i = pt.f0 + k;
                    df g[3];
                    gather_df(M, R, rowptr, sh, pt, k, Pl, cur, b, g[0], g[1], g[2]);
                    fg[i] = g[0].hi; fg[n + i] = g[1].hi; fg[2 * n + i] = g[2].hi;
                }
                cl.sync();
                // back to FP32 reference positions and zero increments
                for (int k = threadIdx.x; k < m; k += blockDim.x) {
                    const int i = pt.gidx(k);
                    float xr[3];
                    for (int c = 0; c < 3; ++c)
                        xr[c] = df_add({Xh[c * n + i], Xl[c * n + i]}, {uh[c * n + i], ul[c * n + i]}).hi;
                    Pl[k] = make_float4(xr[0], xr[1], xr[2], 0.f);
                    cur[k] = make_float4(0.f, 0.f, 0.f, 0.f);
                }
                cl.sync();
                for (int k = grp; k < pt.nfr; k += ngrp) {
                    if (sub != 0) continue;
                    const int i = pt.f0 + k;
                    const float im = imh[i];
                    const float4 va = SV[k];
                    const float g0 = fg[i], g1 = fg[n + i], g2 = fg[2 * n + i];
                    const float a0 = g0 * im - cf * va.x, a1 = g1 * im - cf * va.y,
                                a2 = g2 * im - cf * va.z;
                    const float w0 = va.x + hdtf * a0, w1 = va.y + hdtf * a1, w2 = va.z + hdtf * a2;
                    next_increment(w0, w1, w2, a0, a1, a2, cur[k], hdtf, dtf, SV[k], SA[k], Qb[bn][k]);
                    rs += g0 * g0 + g1 * g1 + g2 * g2;
                    if (want_k) kes += 0.5f * (w0 * w0 + w1 * w1 + w2 * w2) / im;
                }
                since = 0;
            } else {
                vpend = tnow; veval = teval; vbuf = tbuf;
                // L lanes share a node's edges (lane s takes edges s, s+L, ...,
                // two at a time) and combine with shuffles; L is fixed per RVE
                // so its result does not depend on the launch it runs in.
                for (int kb = 0; kb < pt.nfr; kb += ngrp) {
                    const int k = kb + grp;
                    const bool valid = k < pt.nfr;
                    float g0 = 0.f, g1 = 0.f, g2 = 0.f;
                    if (valid) {
                        const float4 qi = cur[k];
                        const int i = pt.f0 + k;
                        const float4 pi = Pl[k];
                        const int end = rowptr[i + 1];
                        int e = rowptr[i] + sub;
                        for (; e + L < end; e += 2 * L) {
                            const int ca = __ldg(colp + e), cb = __ldg(colp + e + L);
                            const float2 ea = __ldg(eafp + e), eb = __ldg(eafp + e + L);
                            const int ra = ca >> 16, la = ca & 0xffff, rb2 = cb >> 16, lb = cb & 0xffff;
                            const float4 pa = ra == pt.me ? Pl[la] : sh.P[ra][la];
                            const float4 qa = ra == pt.me ? cur[la] : sh.Q[b][ra][la];
                            const float4 pb = rb2 == pt.me ? Pl[lb] : sh.P[rb2][lb];
                            const float4 qb = rb2 == pt.me ? cur[lb] : sh.Q[b][rb2][lb];
                            edge_increment(pi, qi, pa, qa, ea, g0, g1, g2);
                            edge_increment(pi, qi, pb, qb, eb, g0, g1, g2);
                        }
                        if (e < end) {
                            const int ca = __ldg(colp + e);
                            const float2 ea = __ldg(eafp + e);
                            const int ra = ca >> 16, la = ca & 0xffff;
                            const float4 pa = ra == pt.me ? Pl[la] : sh.P[ra][la];
                            const float4 qa = ra == pt.me ? cur[la] : sh.Q[b][ra][la];
                            edge_increment(pi, qi, pa, qa, ea, g0, g1, g2);
                        }
                    }
                    for (int o = 1; o < L; o <<= 1) {
                        g0 += __shfl_xor_sync(0xffffffffu, g0, o);
                        g1 += __shfl_xor_sync(0xffffffffu, g1, o);
                        g2 += __shfl_xor_sync(0xffffffffu, g2, o);
                    }
                    if (valid && sub == 0) {
                        const int i = pt.f0 + k;
                        g0 += fg[i]; g1 += fg[n + i]; g2 += fg[2 * n + i];
                        const float im = imh[i];
                        const float4 va = SV[k];
                        float w0 = va.x, w1 = va.y, w2 = va.z;
                        const float a0 = g0 * im - cf * w0;
                        const float a1 = g1 * im - cf * w1;
                        const float a2 = g2 * im - cf * w2;
                        w0 += hdtf * a0; w1 += hdtf * a1; w2 += hdtf * a2;
                        next_increment(w0, w1, w2, a0, a1, a2, cur[k], hdtf, dtf, SV[k], SA[k],
                                       Qb[bn][k]);
                        rs += g0 * g0 + g1 * g1 + g2 * g2;
                        if (want_k) kes += 0.5f * (w0 * w0 + w1 * w1 + w2 * w2) / im;
                    }
                }
            }
            // this evaluation's partials are published in the next barrier's window
            part_rs = rs;
            part_ke = kes;
            part_b = b;
            ++since;
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
    const float4 *Qfin = fin >= 0 ? Qb[fin] : nullptr;
    mixed_finish(cl, sh, M, S, O, P, p, R, pt, F, fin >= 0, [&](int k) { return Qfin[k]; }, status, it, r2, k2, f_ref);
}

}  // namespace

__global__ void __launch_bounds__(512, 1) dr_mixed_plain_lead_kernel(DevMesh M, DevState S, DevResults O,
                                                                     SolveParams P, int part_cap) {
    extern __shared__ __align__(16) float4 dsm[];
    __shared__ MixedShared sh;
    cg::cluster_group cl = cg::this_cluster();
    float4 *Pl = dsm, *Q0 = dsm + part_cap;
    float4 *Qb[kBufs];
    for (int b = 0; b < kBufs; ++b) Qb[b] = Q0;
    map_remote(cl, sh, Pl, Qb, (int)cl.num_blocks());
    int rb = 0;
    for (;;) {
        const int item = next_item(cl, sh, P.counter + (P.resume ? 2 : 0));
        if (item >= P.queue_len) return;
        lead_rve(cl, sh, M, S, O, P, P.queue[item], Pl, Q0, rb);
    }
}

__global__ void __launch_bounds__(512, 1) dr_mixed_fp32_kernel(DevMesh M, DevState S, DevResults O,
                                                               SolveParams P, int part_cap) {
    extern __shared__ __align__(16) float4 dsm[];
    __shared__ MixedShared sh;
    cg::cluster_group cl = cg::this_cluster();
    float4 *Pl = dsm;
    float4 *Qb[kBufs];
    for (int b = 0; b < kBufs; ++b) Qb[b] = dsm + (1 + b) * part_cap;
    map_remote(cl, sh, Pl, Qb, (int)cl.num_blocks());
    for (;;) {
        const int item = next_item(cl, sh, P.counter + 1);
        if (item >= P.queue_len) return;
        fp32_rve(cl, sh, M, S, O, P, P.queue[item], Pl, Qb);
    }
}

namespace {
cudaLaunchConfig_t mixed_config(int clusters, int parts, int block, size_t smem,
                                cudaLaunchAttribute *attr, cudaStream_t st) {
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
std::mutex g_prep_mutex;
std::map<std::pair<const void *, int>, int> g_prep_bytes;  // (kernel, device) -> limit set

template <class K>
void prepare(K kernel, size_t smem) {
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lock(g_prep_mutex);
    int &have = g_prep_bytes[{reinterpret_cast<const void *>(kernel), dev}];
    if (have < (int)smem || have == 0) {
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        have = std::max(have, (int)smem);
    }
}
}  // namespace

// Footprint rule of the cluster size: a part's node state (120 B per node) and
// 52 B per element of its rows within the limit. This is the size of an earlier
// FP32 kernel; dr_mixed_node.cu's, whose row tables are then wholly in shared memory,
// needs less. The rule stays because it sets an RVE's parts, CTA sizes and (parts
// beyond it) order of fused operations: another one would change the trajectories.
size_t mixed_fp32_smem(int part_cap, int free_cap, int elem_cap, int slot_cap, size_t limit) {
    const size_t plain = kFp32PlainNodeBytes * (size_t)part_cap;
    const size_t F = (size_t)free_cap, U = (size_t)elem_cap, S = (size_t)slot_cap;
    const size_t staged = align16(align16(kFp32NodeBytes * (size_t)part_cap) + 16 * F + 3 * 16 * U +
                                  4 * U + 4 * S + 2 * 4 * F + 4 * (F / 32 + 2));
    return staged <= limit ? staged : plain;
}

// Footprint rule of the lead: the staged form (dr_mixed_lead.cu, STAGED) when a
// part's displacements, state and element records are within the limit by this
// count. It is an earlier lead kernel's size too (the present one needs less: 109 KB
// at 800 nodes on one CTA, 187 KB at 1250 on each of 16) and stays for the same
// reason: the form decides the CTA size, the order of the residual's sum and the
// evaluation at which the lead ends.
size_t mixed_lead_smem(int part_cap, int free_cap, int elem_cap, int slot_cap, size_t limit) {
    const size_t plain = kLeadPlainNodeBytes * (size_t)part_cap;
    const size_t F = (size_t)free_cap, U = (size_t)elem_cap, S = (size_t)slot_cap;
    const size_t staged =
        align16(2 * plain + 3 * 16 * F + 4 * 16 * U + 8 * U + 4 * S + 2 * 4 * F + 4 * (F / 32 + 2));
    return staged <= limit ? staged : plain;
}

bool mixed_staged(int lead, size_t smem, int part_cap) {
    return smem > (lead ? kLeadPlainNodeBytes : kFp32PlainNodeBytes) * (size_t)part_cap;
}

size_t mixed_plain_node_bytes(int lead) { return lead ? kLeadPlainNodeBytes : kFp32PlainNodeBytes; }

int launch_dr_mixed(const DevMesh &m, const DevState &s, const DevResults &r, const SolveParams &p,
                    int lead, int clusters, int parts, int block, size_t smem, int part_cap, void *stream) {
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = mixed_config(clusters, parts, block, smem, attr, static_cast<cudaStream_t>(stream));
    const auto kernel = lead ? dr_mixed_plain_lead_kernel : dr_mixed_fp32_kernel;
    prepare(kernel, smem);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, m, s, r, p, part_cap);
    if (e != cudaSuccess) return (int)e;
    return (int)cudaGetLastError();
}

int occupancy_dr_mixed(int lead, int parts, int block, size_t smem) {
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = mixed_config(parts * 64, parts, block, smem, attr, nullptr);
    const auto kernel = lead ? dr_mixed_plain_lead_kernel : dr_mixed_fp32_kernel;
    prepare(kernel, smem);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

}  // namespace fe2
