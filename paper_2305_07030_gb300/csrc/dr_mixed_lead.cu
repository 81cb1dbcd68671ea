// Lead phase of the mixed solver: set-up of an RVE (Algorithm 1 up to the loop)
// and its double-float iterations, one thread-block cluster per RVE. Also the
// resume launch, which finishes RVEs handed back by the FP32 phase.
//
// Arithmetic: displacement form, df_entry_force's operations in its order
// (dr_mixed.cuh). What bounds it is FP32 issue, about 420 instructions per element
// and 600 per node. (The packed .f32x2 instructions take two cycles of the same
// pipe each, and three with distinct registers: 6 % slower here.)
//
// Layout. Each element with an end among a CTA's free nodes has a slot in the
// CTA's table (the batch layout's slots) and is evaluated once per iteration by
// one thread; each free node's thread then sums the +- slot forces of its row in
// row order and moves the node. The displacement array of a CTA holds its own
// free nodes, a copy of each free neighbour in another CTA, which the neighbour's
// thread writes (st.shared::cluster) when it moves its node, and a copy of every
// fixed neighbour, which never changes. The element loop therefore reads its own
// shared memory only.
//
// STAGED (parts that meet the footprint rule): two displacement arrays, one
// cluster barrier per iteration; the next move follows the node's update. The
// last warp evaluates no elements: it adds and judges residuals while the others
// do. The verdict on evaluation n is known three evaluations later, and the lead
// ends there. With KSM the element constants are in shared memory, else they are
// read from the batch's arrays (L2).
// !STAGED (larger parts): one displacement array, velocity and acceleration in
// global memory, every evaluation judged before the next move.
//
// Measured against the kernels it replaced (one more pass per iteration for the
// move, the testing warp ahead of its own elements, the far ends' displacements
// read across the cluster; without a table, rows re-read from L2 and each element
// evaluated from both ends): 64 RVEs of 5000 nodes x 400 iterations 12.6 -> 11.2
// ms, 256 of 1000 x 200 4.35 -> 3.98, 8 of 37 to 200 x 100 0.31 -> 0.25, 24 of
// 1k to 33k x 200 10.3 -> 6.9 (the parts without a table), and the one-part RVEs
// of 780 to about 820 nodes, which had none either, 22.2 -> 8.3 us per iteration (790 nodes).
#include <algorithm>
#include <map>
#include <mutex>
#include <type_traits>
#include <utility>

#include "dr_mixed.cuh"

namespace fe2 {

namespace {

struct LeadShared : ResidualSums {
    Verdict vd[2];                      // by evaluation parity
    double sig[kMaxParts][9];           // stress partials, read by rank 0
    double wsum[kMaxWarps][9];
    double *sigp;                       // rank 0's sig
    int item;
};

// Tables of one CTA (shared memory; lead_smem gives the layout). A displacement
// or velocity is (x.hi, y.hi, x.lo, y.lo) and (z.hi, z.lo), a force likewise.
struct LeadTables {
    float4 *UA;    // displacements: one array of u_cap, two with STAGED
    float4 *TA;    // per slot: force on the element's first end
    float4 *K0;    // KSM, per slot: (D, L).hi, D = X_second - X_first
    float4 *K1;    // (D, L).lo
    float4 *VA;    // STAGED, per own free node: half-step velocity
    float2 *UB, *TB, *VB;
    float2 *KA;    // KSM, per slot: EA/L
    float2 *IM;    // STAGED, per own free node: 1/m
    uint32_t *EN;  // KSM, per slot: places of its ends in the displacement array
    uint32_t *PA;  // copies of own nodes: part << 16 | place in its displacement array
    uint32_t *PO;  // per own free node: first copy | count << 24
    int *SS;       // per slab + 1: first row entry
    uint16_t *NS;  // per row entry: slot << 1 | 1 if the node is the second end
    uint16_t *RL;  // per own free node: row length
};

struct Node {  // a double-float vector
    df x, y, z;
};
__device__ __forceinline__ Node node_load(const float4 &a, const float2 &b) {
    return {{a.x, a.z}, {a.y, a.w}, {b.x, b.y}};
}
__device__ __forceinline__ void node_store(const Node &n, float4 &a, float2 &b) {
    a = make_float4(n.x.hi, n.y.hi, n.x.lo, n.y.lo);
    b = make_float2(n.z.hi, n.z.lo);
}
__device__ __forceinline__ Node node_read(const float *h, const float *l, int n, int i) {
    return {{h[i], l[i]}, {h[n + i], l[n + i]}, {h[2 * n + i], l[2 * n + i]}};
}
__device__ __forceinline__ void node_write(const Node &v, float *h, float *l, int n, int i) {
    h[i] = v.x.hi; h[n + i] = v.y.hi; h[2 * n + i] = v.z.hi;
    l[i] = v.x.lo; l[n + i] = v.y.lo; l[2 * n + i] = v.z.lo;
}
__device__ __forceinline__ Node node_add(const Node &a, const Node &b) {
    return {df_add(a.x, b.x), df_add(a.y, b.y), df_add(a.z, b.z)};
}
__device__ __forceinline__ Node node_sub(const Node &a, const Node &b) {
    return {df_sub(a.x, b.x), df_sub(a.y, b.y), df_sub(a.z, b.z)};
}
__device__ __forceinline__ Node node_scale(const Node &a, df s) { return {df_mul(a.x, s), df_mul(a.y, s), df_mul(a.z, s)}; }
// s a, with the scalar as the first factor
__device__ __forceinline__ Node scale_node(df s, const Node &a) { return {df_mul(s, a.x), df_mul(s, a.y), df_mul(s, a.z)}; }

// Force on the first end of an element with displacements u, w of its ends, (D, L)
// and EA/L: the operations of df_entry_force.
__device__ __forceinline__ Node element_force(const Node &u, const Node &w, const float4 &Dh, const float4 &Dl,
                                              const float2 &kx) {
    const Node e = node_sub(w, u);
    const Node D = {{Dh.x, Dl.x}, {Dh.y, Dl.y}, {Dh.z, Dl.z}};
    const df L = {Dh.w, Dl.w};
    const Node d = node_add(D, e), b = node_add(D, d);
    const df h = df_add(df_add(df_mul(e.x, b.x), df_mul(e.y, b.y)), df_mul(e.z, b.z));
    const df l2 = df_add(df_sqr(L), h);
    const df rl = df_rsqrt(l2);
    const df l = df_mul(l2, rl);
    const df q = df_mul(df_mul({kx.x, kx.y}, df_mul(h, rl)), df_rcp(df_add(l, L)));
    return scale_node(q, d);
}

// Constants of slot u from the batch's arrays: w = CSR entry << 1 | 1 when the
// entry runs from the second end to the first.
__device__ __forceinline__ void slot_constants(const DevMesh &M, const RveDesc &R, int w, float4 &Dh, float4 &Dl,
                                               float2 &kx) {
    const int64_t kk = R.csr0 + (w >> 1);
    Dh = M.dh[kk];
    Dl = M.dl[kk];
    if (w & 1) {
        Dh.x = -Dh.x; Dh.y = -Dh.y; Dh.z = -Dh.z;
        Dl.x = -Dl.x; Dl.y = -Dl.y; Dl.z = -Dl.z;
    }
    const float2 eh = M.eaf[kk], el = M.eaf_lo[kk];
    const df k = df_mul({eh.x, el.x}, {eh.y, el.y});
    kx = make_float2(k.hi, k.lo);
}

// Double-float internal force on node i from displacements in global memory.
__device__ __noinline__ void lead_gather(const DevMesh &M, const RveDesc &R, const float *uh, const float *ul, int i,
                                         df *g) {
    const int n = R.n_nodes;
    const int32_t *rowptr = M.rowptr + R.rp0;
    const df ui0 = {uh[i], ul[i]}, ui1 = {uh[n + i], ul[n + i]}, ui2 = {uh[2 * n + i], ul[2 * n + i]};
    df g0 = df_from(0.f), g1 = df_from(0.f), g2 = df_from(0.f);
    for (int e = rowptr[i]; e < rowptr[i + 1]; ++e) {
        const int64_t kk = R.csr0 + e;
        const int j = M.col[kk];
        df_entry_force(M, kk, df_sub({uh[j], ul[j]}, ui0), df_sub({uh[n + j], ul[n + j]}, ui1),
                       df_sub({uh[2 * n + j], ul[2 * n + j]}, ui2), g0, g1, g2);
    }
    g[0] = g0; g[1] = g1; g[2] = g2;
}

// Square root of the cluster's sum of one value per thread (set-up).
__device__ __forceinline__ double lead_norm(LeadShared &sh, float acc, int me, int C) {
    sh.rs[0][threadIdx.x >> 5][threadIdx.x & 31] = acc;
    __syncthreads();
    if ((int)(threadIdx.x >> 5) == (int)(blockDim.x >> 5) - 1) publish_sums(sh, 0, 0, me, C, false);
    cg::this_cluster().sync();
    const Verdict v = sums_verdict(sh, 0, C, df_from(0.f), 0, false, INT64_MAX);
    cg::this_cluster().sync();
    return sqrt(df_to_double({v.r2h, v.r2l}));
}

// Initial displacement, velocity and acceleration into the state arrays;
// returns f_ref. With the affine start both reference forces are the same.
__device__ __noinline__ double lead_start(LeadShared &sh, const DevMesh &M, const DevState &S, const SolveParams &P,
                                          int p, const RveDesc &R, const Part pt, bool staged) {
    const int n = R.n_nodes, m = pt.m();
    const int64_t n0 = R.node0, b3 = 3 * n0;
    float *uh = S.uh + b3, *ul = S.ul + b3, *vh = S.vh + b3, *vl = S.vl + b3;
    float *ah = S.ah + b3, *al = S.al + b3, *fg = S.fg + b3;
    double F[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) F[k] = P.F[9 * (int64_t)p + k];
    // affine displacement (F - I) X, in the velocity arrays until its force is
    // known, and the initial one
    for (int k = threadIdx.x; k < m; k += blockDim.x) {
        const int i = pt.gidx(k);
        const double X[3] = {M.X0[n0 + i], M.X1[n0 + i], M.X2[n0 + i]};
        const double *uw[3] = {S.u0 + n0, S.u1 + n0, S.u2 + n0};
        for (int r = 0; r < 3; ++r) {
            const double xa = dadd(dadd(dmul(F[3 * r], X[0]), dmul(F[3 * r + 1], X[1])), dmul(F[3 * r + 2], X[2]));
            const double uaff = dsub(xa, X[r]);
            const double u = k >= pt.nfr || P.init == 1 ? uaff : P.init == 2 ? uw[r][i] : 0.0;
            const df ud = df_from_double(u), ua = df_from_double(uaff);
            uh[r * n + i] = ud.hi;
            ul[r * n + i] = ud.lo;
            vh[r * n + i] = ua.hi;
            vl[r * n + i] = ua.lo;
        }
    }
    cg::this_cluster().sync();
    // |g|^2 in the two orders of its fused products: parts beyond the footprint rule
    // have always summed the affine force's (AFF) and the initial force's in different
    // ones; they keep them (and an affine start its second sum) only for f_ref's bits.
    auto square = [&](const df *g, bool aff) {
        const float x = g[0].hi, y = g[1].hi, z = g[2].hi;
        return aff && !staged ? dot3(y, x, z, y, x, z) : dot3(x, y, z, x, y, z);
    };
    double f_aff = 0.0;
    df g[3];
    float acc = 0.f, acc_aff = 0.f;
    if (P.init != 1) {
        for (int k = threadIdx.x; k < m; k += blockDim.x) {
            lead_gather(M, R, vh, vl, pt.gidx(k), g);
            acc_aff = fadd(acc_aff, square(g, true));
        }
        f_aff = lead_norm(sh, acc_aff, pt.me, pt.C);
    }
    for (int k = threadIdx.x; k < m; k += blockDim.x) {
        const int i = pt.gidx(k);
        lead_gather(M, R, uh, ul, i, g);
        acc = fadd(acc, square(g, false));
        if (P.init == 1) acc_aff = fadd(acc_aff, square(g, true));
        if (k < pt.nfr) {
            const df im = {M.imh[n0 + i], M.iml[n0 + i]};
            for (int r = 0; r < 3; ++r) {
                const df a = df_mul(g[r], im);
                ah[r * n + i] = a.hi;
                al[r * n + i] = a.lo;
                vh[r * n + i] = 0.f;
                vl[r * n + i] = 0.f;
                fg[r * n + i] = g[r].hi;
            }
        }
    }
    if (P.init == 1 && !staged) f_aff = lead_norm(sh, acc_aff, pt.me, pt.C);
    const double f0 = lead_norm(sh, acc, pt.me, pt.C);
    return f_aff > f0 ? f_aff : f0;
}

struct NoInc {  // no FP32 increment on top of the double-float displacement
    __device__ float4 operator()(int) const { return make_float4(0.f, 0.f, 0.f, 0.f); }
};
__device__ __noinline__ void lead_finish(LeadShared &sh, const DevMesh &M, const DevState &S, const DevResults &O,
                                         const SolveParams &P, int p, const RveDesc &R, const Part pt, int status,
                                         int64_t it, df r2, df k2, double f_ref) {
    cg::cluster_group cl = cg::this_cluster();
    double F[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) F[k] = P.F[9 * (int64_t)p + k];
    mixed_finish(cl, sh, M, S, O, P, p, R, pt, F, false, NoInc{}, status, it, r2, k2, f_ref);
}

// Iterations from the state arrays at evaluation `it`, until the lead's end
// (lead2, lead_iters), convergence, NaN or max_iter; the state goes back to the
// arrays, with the reference force of the last evaluation.
template <bool STAGED, bool KSM>
__device__ __forceinline__ void lead_loop(LeadShared &sh, const DevMesh &M, const DevState &S, const RveDesc &R,
                                          const Part &pt, const SolveParams &P, const LeadShape &sp,
                                          const LeadTables &T, int64_t lead_iters, df lead2, df thresh2, df dt, df hdt,
                                          df cdf, int64_t &it, int &status, df &r2, df &k2) {
    cg::cluster_group cl = cg::this_cluster();
    const int64_t it0 = it;
    const int n = R.n_nodes, nfr = pt.nfr, C = sp.parts, p = (int)(&R - M.rve);
    const int64_t n0 = R.node0, b3 = 3 * n0;
    float *uh = S.uh + b3 + pt.f0, *ul = S.ul + b3 + pt.f0, *vh = S.vh + b3 + pt.f0, *vl = S.vl + b3 + pt.f0;
    float *ah = S.ah + b3 + pt.f0, *al = S.al + b3 + pt.f0, *fg = S.fg + b3 + pt.f0;
    const float *imh = M.imh + n0 + pt.f0, *iml = M.iml + n0 + pt.f0;
    const bool want_k = P.want_ke != 0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // The first slabs have the longest rows: every other four warps (one per
    // scheduler) take theirs in reverse, which evens the schedulers' node work.
    const int nslot = (blockDim.x & 127u) == 0 && (warp & 4) ? warp ^ 3 : warp;
    const int k0 = 32 * nslot + lane;
    const int W = (int)blockDim.x - 32;  // the element threads
    const bool test_warp = (int)threadIdx.x >= W;
    const int32_t *ps = M.ls_part_slot + (int64_t)p * (kMaxParts + 1);
    const int s0 = ps[pt.me], n_el = ps[pt.me + 1] - s0;
    const int4 *slots = M.ls_slot + R.ls_slot0 + s0;
    const uint32_t *ends = M.lead_ends + R.ls_slot0 + s0;

    // ---- tables ----
    {
        const int32_t *frow = M.ls_row + R.rp0 + pt.f0, *fent = M.ls_csr_slot + R.csr0;
        slab_offsets(T.SS, nfr, [&](int k) { return frow[k + 1] - frow[k]; });
        copy_lists(M, R, pt, T.PO, [&](int x, uint32_t w) { T.PA[x] = w; });
        const int32_t *fo = M.lead_fix_off + (int64_t)p * 2 * (kMaxParts + 1);
        const int f0 = fo[pt.me], nf = fo[pt.me + 1] - f0, at = fo[kMaxParts + 1 + pt.me];
        for (int k = threadIdx.x; k < nf; k += blockDim.x) {
            const int i = M.lead_fix[R.fix0 + f0 + k];
            const Node u = node_read(S.uh + b3, S.ul + b3, n, i);
            for (int t = 0; t < (STAGED ? 2 : 1); ++t)
                node_store(u, T.UA[t * sp.u_cap + at + k], T.UB[t * sp.u_cap + at + k]);
        }
        if (KSM)
            for (int u = threadIdx.x; u < n_el; u += blockDim.x) {
                slot_constants(M, R, slots[u].w, T.K0[u], T.K1[u], T.KA[u]);
                T.EN[u] = ends[u];
            }
        __syncthreads();
        for (int k = threadIdx.x; k < nfr; k += blockDim.x) {
            const int beg = frow[k], deg = frow[k + 1] - beg;
            int sl = T.SS[k >> 5] + (k & 31);
            T.RL[k] = (uint16_t)deg;
            for (int e = 0; e < deg; ++e, sl += 32) T.NS[sl] = (uint16_t)fent[beg + e];
        }
    }
    // Move own node k to the next evaluation: v += dt/2 a, u += dt v; u and its
    // copies into array t.
    auto move = [&](int k, Node &v, const Node &a, const Node &u, int t) {
        v = node_add(v, scale_node(hdt, a));
        const Node x = node_add(u, scale_node(dt, v));
        float4 A;
        float2 B;
        node_store(x, A, B);
        const int at = t * sp.u_cap;
        T.UA[at + k] = A;
        T.UB[at + k] = B;
        const uint32_t po = T.PO[k], ua = smem_addr(T.UA + at), ub = smem_addr(T.UB + at);
        for (uint32_t c = po & 0xffffffu, e = c + (po >> 24); c < e; ++c) {
            const uint32_t w = T.PA[c], q = w & 0xffffu;
            st_cluster(cluster_addr(ua + 16u * q, w >> 16), A);
            st_cluster(cluster_addr(ub + 8u * q, w >> 16), B);
        }
    };
    // Element forces of array t: slots u, u + step, ... two at a time (a chain
    // is about 800 cycles of latency).
    auto batch = [&](int t, int u0, int step, auto count) {
        constexpr int N = decltype(count)::value;
        const float4 *UA = T.UA + t * sp.u_cap;
        const float2 *UB = T.UB + t * sp.u_cap;
        Node a[N], b[N];
        float4 Dh[N], Dl[N];
        float2 kx[N];
#pragma unroll
        for (int x = 0; x < N; ++x) {
            const int u = u0 + x * step;
            const uint32_t w = KSM ? T.EN[u] : ends[u], i = w & 0xffffu, j = w >> 16;
            a[x] = node_load(UA[i], UB[i]);
            b[x] = node_load(UA[j], UB[j]);
            if (KSM) {
                Dh[x] = T.K0[u];
                Dl[x] = T.K1[u];
                kx[x] = T.KA[u];
            } else {
                slot_constants(M, R, slots[u].w, Dh[x], Dl[x], kx[x]);
            }
        }
#pragma unroll
        for (int x = 0; x < N; ++x)
            node_store(element_force(a[x], b[x], Dh[x], Dl[x], kx[x]), T.TA[u0 + x * step], T.TB[u0 + x * step]);
    };
    auto elements = [&](int t, int first, int step) {
        int u = first;
        for (; u + step < n_el; u += 2 * step) batch(t, u, step, std::integral_constant<int, 2>());
        if (u < n_el) batch(t, u, step, std::integral_constant<int, 1>());
    };
    // Row sum of own node k, in row order (the second end receives -t); two
    // entries' loads at a time.
    auto entry = [&](int sl) {
        const uint32_t e = T.NS[sl], sg = (e & 1u) << 31;
        const float4 a = T.TA[e >> 1];
        const float2 b = T.TB[e >> 1];
        auto flip = [&](float x) { return __uint_as_float(__float_as_uint(x) ^ sg); };
        return node_load(make_float4(flip(a.x), flip(a.y), flip(a.z), flip(a.w)), make_float2(flip(b.x), flip(b.y)));
    };
    auto gather = [&](int k) {
        int w = T.RL[k], sl = T.SS[k >> 5] + (k & 31);
        Node g = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
        for (; w >= 2; w -= 2, sl += 64) {
            const Node f0 = entry(sl), f1 = entry(sl + 32);
            g = node_add(node_add(g, f0), f1);
        }
        if (w > 0) g = node_add(g, entry(sl));
        return g;
    };
    // Acceleration and full-step velocity (Algorithm 1: damping, a = (g + f_d)/m,
    // v += dt/2 a), residual and kinetic-energy terms.
    auto update = [&](const Node &g, df im, Node &v, Node &a, float &rs, float &kes) {
        a = node_sub(node_scale(g, im), scale_node(cdf, v));
        v = node_add(v, scale_node(hdt, a));
        rs = __fmaf_rn(g.z.hi, g.z.hi, __fmaf_rn(g.y.hi, g.y.hi, __fmaf_rn(g.x.hi, g.x.hi, rs)));
        if (!want_k) return;
        const float vv = __fmaf_rn(v.z.hi, v.z.hi, __fmaf_rn(v.y.hi, v.y.hi, __fmaf_rn(v.x.hi, v.x.hi, 0.f)));
        kes = fadd(kes, __fdiv_rn(fmul(0.5f, vv), im.hi));
    };
    auto write_fg = [&](int k, const Node &g) {
        fg[k] = g.x.hi; fg[n + k] = g.y.hi; fg[2 * n + k] = g.z.hi;
    };

    // the first move
    for (int k = k0; k < nfr; k += blockDim.x) {
        Node v = node_read(vh, vl, n, k);
        const Node a = node_read(ah, al, n, k), u = node_read(uh, ul, n, k);
        move(k, v, a, u, STAGED ? (int)((it + 1) & 1) : 0);
        if (STAGED) {
            node_store(v, T.VA[k], T.VB[k]);
            T.IM[k] = make_float2(imh[k], iml[k]);
        } else {
            node_write(v, vh, vl, n, k);
        }
    }
    Verdict v = {-1, 0.f, 0.f, 0.f, 0.f};
    for (;;) {
        ++it;  // this iteration's evaluation
        const int t = STAGED ? (int)(it & 1) : 0, sb = (int)(it % 3);
        if (C > 1) {
            cluster_arrive();
            cluster_wait();
        } else {
            __syncthreads();
        }
        float rs = 0.f, kes = 0.f;
        if (STAGED) {
            // the verdict on evaluation it - 3 decides whether this one is the last
            const int code = it >= it0 + 4 ? sh.vd[t ^ 1].code : -1;
            const bool last = code == RVE_NAN || it >= P.max_iter || (lead_iters >= 0 ? it >= lead_iters : code == RVE_OK);
            if (!test_warp) {
                elements(t, threadIdx.x, W);
            } else {
                // sums of evaluation it - 1, verdict on evaluation it - 2
                if (it >= it0 + 3) {
                    const Verdict mine = sums_verdict(sh, (int)((it - 2) % 3), C, lead2, 0, want_k, INT64_MAX);
                    if (lane == 0) sh.vd[t] = mine;
                }
                if (it >= it0 + 2) publish_sums(sh, t ^ 1, (int)((it - 1) % 3), pt.me, C, want_k);
            }
            __syncthreads();
            for (int k = k0; k < nfr; k += blockDim.x) {
                const Node g = gather(k);
                Node vk = node_load(T.VA[k], T.VB[k]), a;
                update(g, {T.IM[k].x, T.IM[k].y}, vk, a, rs, kes);
                const Node u = node_load(T.UA[t * sp.u_cap + k], T.UB[t * sp.u_cap + k]);
                if (!last) {
                    move(k, vk, a, u, t ^ 1);
                    node_store(vk, T.VA[k], T.VB[k]);
                } else {
                    write_fg(k, g);
                    node_write(u, uh, ul, n, k);
                    node_write(vk, vh, vl, n, k);
                    node_write(a, ah, al, n, k);
                }
            }
            sh.rs[t][nslot][lane] = rs;
            if (want_k) sh.ke[t][nslot][lane] = kes;
            if (!last) continue;
            // the hand-over evaluation's own residual
            __syncthreads();
            if (test_warp) publish_sums(sh, t, sb, pt.me, C, want_k);
            cl.sync();
            v = sums_verdict(sh, sb, C, thresh2, it, want_k, P.max_iter);
            break;
        } else {
            elements(0, threadIdx.x, blockDim.x);
            __syncthreads();
            for (int k = k0; k < nfr; k += blockDim.x) {
                const Node g = gather(k);
                Node vk = node_read(vh, vl, n, k), a;
                update(g, {imh[k], iml[k]}, vk, a, rs, kes);
                write_fg(k, g);
                node_write(vk, vh, vl, n, k);
                node_write(a, ah, al, n, k);
            }
            sh.rs[0][nslot][lane] = rs;
            if (want_k) sh.ke[0][nslot][lane] = kes;
            __syncthreads();
            if (test_warp) publish_sums(sh, 0, sb, pt.me, C, want_k);
            if (C > 1) {
                cluster_arrive();
                cluster_wait();
            } else {
                __syncthreads();
            }
            v = sums_verdict(sh, sb, C, thresh2, it, want_k, P.max_iter);
            if (v.code >= 0 || (lead_iters >= 0 ? it >= lead_iters : df_le({v.r2h, v.r2l}, lead2))) break;
            for (int k = k0; k < nfr; k += blockDim.x) {
                Node vk = node_read(vh, vl, n, k);
                move(k, vk, node_read(ah, al, n, k), node_load(T.UA[k], T.UB[k]), 0);
                node_write(vk, vh, vl, n, k);
            }
        }
    }
    if (!STAGED)
        for (int k = k0; k < nfr; k += blockDim.x) node_write(node_load(T.UA[k], T.UB[k]), uh, ul, n, k);
    r2 = {v.r2h, v.r2l};
    k2 = {v.k2h, v.k2l};
    status = v.code >= 0 ? v.code : RVE_PENDING;
    cl.sync();  // the tables may be rebuilt
}

template <bool STAGED, bool KSM>
__device__ __forceinline__ void lead_rve(LeadShared &sh, const DevMesh &M, const DevState &S, const DevResults &O,
                                         const SolveParams &P, const LeadShape &sp, int p, const LeadTables &T) {
    cg::cluster_group cl = cg::this_cluster();
    const RveDesc &R = M.rve[p];
    const Part pt = make_part(M, R, p, (int)cl.block_rank(), sp.parts);
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
    } else {
        f_ref = lead_start(sh, M, S, P, p, R, pt, STAGED);
    }
    const df thresh2 = df_from_double(dmul(dmul(P.tol, f_ref), dmul(P.tol, f_ref)));
    // a resumed RVE runs in double-float until it converges
    const df lead2 = P.resume ? thresh2 : df_from_double(dmul(dmul(P.lead_tol, f_ref), dmul(P.lead_tol, f_ref)));
    const int64_t lead_iters = P.resume ? -1 : P.lead_iters;
    const double dt64 = dmul(P.alpha, R.dtc);
    const df dt = df_from_double(dt64), hdt = df_from_double(dmul(0.5, dt64)), cdf = df_from_double(R.c);
    const int64_t it0 = it;
    int status = RVE_PENDING;
    df r2 = df_from(0.f), k2 = df_from(0.f);
    // The STAGED loop ends three evaluations after the tested one; when resuming,
    // the state it ends at must itself be converged, else it goes on from there.
    do {
        lead_loop<STAGED, KSM>(sh, M, S, R, pt, P, sp, T, lead_iters, lead2, thresh2, dt, hdt, cdf, it, status, r2, k2);
    } while (P.resume && status == RVE_PENDING);
    if (P.resume) {
        if (pt.me == 0 && threadIdx.x == 0) O.lead[p] += it - it0;
        lead_finish(sh, M, S, O, P, p, R, pt, status, it, r2, k2, f_ref);
        return;
    }
    if (pt.me == 0 && threadIdx.x == 0) {
        O.iters[p] = it;
        O.lead[p] = it;
        O.status[p] = status;
        O.f_ref[p] = f_ref;
        O.rel_res[p] = df_to_double(r2);  // squared residual, finished by the FP32 phase
        O.ke[p] = P.want_ke != 0 ? df_to_double(k2) : 0.0;
    }
}

}  // namespace

template <bool STAGED, bool KSM>
__global__ void __launch_bounds__(512, 1)
    dr_mixed_lead_kernel(const __grid_constant__ DevMesh M, const __grid_constant__ DevState S,
                         const __grid_constant__ DevResults O, const __grid_constant__ SolveParams P,
                         const __grid_constant__ LeadShape sp) {
    extern __shared__ __align__(16) float4 dsm_lead[];
    __shared__ __align__(16) LeadShared sh;
    cg::cluster_group cl = cg::this_cluster();
    constexpr int A = STAGED ? 2 : 1;
    LeadTables T = {};
    // layout as in lead_smem
    T.UA = dsm_lead;
    T.TA = T.UA + A * sp.u_cap;
    float4 *q = T.TA + sp.elem_cap;
    if (KSM) {
        T.K0 = q;
        T.K1 = T.K0 + sp.elem_cap;
        q = T.K1 + sp.elem_cap;
    }
    if (STAGED) {
        T.VA = q;
        q = T.VA + sp.free_cap;
    }
    T.UB = reinterpret_cast<float2 *>(q);
    T.TB = T.UB + A * sp.u_cap;
    float2 *d = T.TB + sp.elem_cap;
    if (KSM) {
        T.KA = d;
        d = T.KA + sp.elem_cap;
    }
    if (STAGED) {
        T.VB = d;
        T.IM = T.VB + sp.free_cap;
        d = T.IM + sp.free_cap;
    }
    uint32_t *w = reinterpret_cast<uint32_t *>(d);
    if (KSM) {
        T.EN = w;
        w = T.EN + sp.elem_cap;
    }
    T.PA = w;
    T.PO = T.PA + sp.push_cap;
    T.SS = reinterpret_cast<int *>(T.PO + sp.free_cap);
    T.NS = reinterpret_cast<uint16_t *>(T.SS + sp.free_cap / 32 + 2);
    T.RL = T.NS + sp.slot_cap;
    if (threadIdx.x == 0) sh.sigp = cl.map_shared_rank(&sh.sig[0][0], 0);
    for (;;) {
        if (cl.block_rank() == 0 && threadIdx.x == 0) sh.item = atomicAdd(P.counter + (P.resume ? 2 : 0), 1);
        cl.sync();
        const int item = *cl.map_shared_rank(&sh.item, 0);
        cl.sync();
        if (item >= P.queue_len) return;
        lead_rve<STAGED, KSM>(sh, M, S, O, P, sp, P.queue[item], T);
    }
}

namespace {
using LeadKernel = void (*)(DevMesh, DevState, DevResults, SolveParams, LeadShape);

LeadKernel pick_lead(const LeadShape &sp) {
    if (!sp.staged) return sp.ksm ? dr_mixed_lead_kernel<false, true> : dr_mixed_lead_kernel<false, false>;
    return sp.ksm ? dr_mixed_lead_kernel<true, true> : dr_mixed_lead_kernel<true, false>;
}

cudaLaunchConfig_t lead_config(int clusters, int block, const LeadShape &sp, cudaLaunchAttribute *attr, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(clusters * sp.parts, 1, 1);
    cfg.blockDim = dim3(block, 1, 1);
    cfg.dynamicSmemBytes = lead_smem(sp);
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = sp.parts;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

// Raise a kernel's dynamic shared-memory limit (and allow 16-CTA clusters)
// once per device and size, so that launches recorded into a CUDA graph make
// no attribute calls of their own.
std::mutex g_lead_mutex;
std::map<std::pair<const void *, int>, int> g_lead_bytes;

void prepare_lead(LeadKernel k, size_t smem) {
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lock(g_lead_mutex);
    int &have = g_lead_bytes[{reinterpret_cast<const void *>(k), dev}];
    if (have == 0 || have < (int)smem) {
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        have = std::max(have, (int)smem);
    }
}
}  // namespace

size_t lead_smem(const LeadShape &sp) {
    const size_t U = (size_t)sp.u_cap * (sp.staged ? 2 : 1), E = (size_t)sp.elem_cap, F = (size_t)sp.free_cap;
    size_t b = 24 * U + 24 * E + (sp.ksm ? 44 * E : 0) + (sp.staged ? 32 * F : 0) + 4 * (size_t)sp.push_cap + 4 * F +
               4 * (F / 32 + 2) + 2 * ((size_t)sp.slot_cap + F);
    return (b + 15) & ~size_t(15);
}

int launch_dr_mixed_lead(const DevMesh &m, const DevState &s, const DevResults &r, const SolveParams &p, int clusters,
                         int block, const LeadShape &sp, void *stream) {
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = lead_config(clusters, block, sp, attr, static_cast<cudaStream_t>(stream));
    const LeadKernel k = pick_lead(sp);
    prepare_lead(k, cfg.dynamicSmemBytes);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k, m, s, r, p, sp);
    if (e != cudaSuccess) return (int)e;
    return (int)cudaGetLastError();
}

int occupancy_dr_mixed_lead(int block, const LeadShape &sp) {
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = lead_config(64, block, sp, attr, nullptr);
    const LeadKernel k = pick_lead(sp);
    prepare_lead(k, cfg.dynamicSmemBytes);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

}  // namespace fe2
