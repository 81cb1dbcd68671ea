// Helpers shared by the mixed-precision kernels (dr_mixed.cu, dr_mixed_lead.cu,
// dr_mixed_node.cu): a part of an RVE, cluster barriers, row tables, the residual
// test and the end of a solve.
#pragma once
#include <cooperative_groups.h>

#include "df64.cuh"
#include "dr_device.cuh"

namespace fe2 {

namespace cg = cooperative_groups;

namespace {

constexpr int kMaxWarps = 16;  // blocks of at most 512 threads
constexpr int kBufs = 5;       // FP32 phase: evaluations whose state and partials are kept

struct Part {
    int me, C;
    int f0, nfr;   // own free nodes: RVE-local [f0, f0 + nfr)
    int g0, nfx;   // own fixed nodes: RVE-local n_free + [g0, g0 + nfx)
    int nf;        // RVE free count
    __device__ int gidx(int k) const { return k < nfr ? f0 + k : nf + g0 + (k - nfr); }
    __device__ int m() const { return nfr + nfx; }
};

__device__ __forceinline__ Part make_part(const DevMesh &M, const RveDesc &R, int p, int me, int C) {
    const int32_t *po = M.part_off + (int64_t)p * 2 * (kMaxParts + 1);
    Part pt;
    pt.me = me;
    pt.C = C;
    pt.nf = R.n_free;
    pt.f0 = po[me];
    pt.nfr = po[me + 1] - pt.f0;
    pt.g0 = po[kMaxParts + 1 + me];
    pt.nfx = po[kMaxParts + 1 + me + 1] - pt.g0;
    return pt;
}

__device__ __forceinline__ void cluster_arrive() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

// Convergence verdict on one evaluation (FP32 kernel): code -1 = go on, else
// the RVE status; the double-float squared residual and kinetic energy.
struct Verdict {
    int code;
    float r2h, r2l, k2h, k2l;
};

// a <= b for double-float values.
__device__ __forceinline__ bool df_le(df a, df b) { return a.hi < b.hi || (a.hi == b.hi && a.lo <= b.lo); }

// 32-bit shared-memory address of p and its image in cluster CTA `rank`.
__device__ __forceinline__ uint32_t smem_addr(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint32_t cluster_addr(uint32_t a, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_cluster(uint32_t a, const float4 &v) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};"
                 :: "r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ void st_cluster(uint32_t a, const float2 &v) {
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" :: "r"(a), "f"(v.x), "f"(v.y) : "memory");
}

// a . b, every rounding explicit.
__device__ __forceinline__ float dot3(float a0, float a1, float a2, float b0, float b1, float b2) {
    return __fmaf_rn(a2, b2, __fmaf_rn(a0, b0, fmul(a1, b1)));
}

// First slot of each slab of 32 rows (ELL: a slab is as wide as its first row, the
// rows are sorted by degree) into SS, by the first warp; deg(k) is a row's length.
template <class Deg>
__device__ __forceinline__ void slab_offsets(int *SS, int nfr, const Deg &deg) {
    const int lane = threadIdx.x & 31, ns = (nfr + 31) >> 5;
    if (threadIdx.x >= 32) return;
    int base = 0;
    for (int s0 = 0; s0 < ns; s0 += 32) {
        const int s = s0 + lane;
        int w = s < ns ? 32 * deg(32 * s) : 0;
        const int own = w;
        for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += x;
        }
        if (s < ns) SS[s] = base + w - own;
        base += __shfl_sync(0xffffffffu, w, 31);
    }
    if (lane == 0) SS[ns] = base;
}

// The copies of this CTA's nodes in other CTAs: set(x, part << 16 | place) for
// each, and, per own free node, first copy | count << 24 into PO.
template <class Set>
__device__ __forceinline__ void copy_lists(const DevMesh &M, const RveDesc &R, const Part &pt, uint32_t *PO,
                                           const Set &set) {
    const int32_t *po = M.push_off + R.rp0 + pt.f0;
    const int p0 = po[0];
    for (int k = threadIdx.x; k < pt.nfr; k += blockDim.x)
        PO[k] = (uint32_t)(po[k] - p0) | ((uint32_t)(po[k + 1] - po[k]) << 24);
    for (int x = threadIdx.x; x < po[pt.nfr] - p0; x += blockDim.x) set(x, M.push[R.push0 + p0 + x]);
}

// Double-float force of CSR entry kk on its row's node in displacement form
// (Algorithm 1, getInternalForces), added to g: e = u_j - u_i, d = D + e, and
// N/l = EA (l - L) / (L l) = (EA/L) h / (l (l + L)), h = l^2 - L^2 = e.(D + d),
// which has no cancellation.
__device__ __forceinline__ void df_entry_force(const DevMesh &M, int64_t kk, df e0, df e1, df e2, df &g0, df &g1,
                                               df &g2) {
    const float4 Dh = M.dh[kk], Dl = M.dl[kk];
    const df D0 = {Dh.x, Dl.x}, D1 = {Dh.y, Dl.y}, D2 = {Dh.z, Dl.z}, L = {Dh.w, Dl.w};
    const df d0 = df_add(D0, e0), d1 = df_add(D1, e1), d2 = df_add(D2, e2);
    const df h = df_add(df_add(df_mul(e0, df_add(D0, d0)), df_mul(e1, df_add(D1, d1))),
                        df_mul(e2, df_add(D2, d2)));
    const df l2 = df_add(df_sqr(L), h);
    const df rl = df_rsqrt(l2);
    const df l = df_mul(l2, rl);
    const float2 eh = M.eaf[kk], el = M.eaf_lo[kk];
    const df kax = df_mul({eh.x, el.x}, {eh.y, el.y});
    const df q = df_mul(df_mul(kax, df_mul(h, rl)), df_rcp(df_add(l, L)));
    g0 = df_add(g0, df_mul(q, d0));
    g1 = df_add(g1, df_mul(q, d1));
    g2 = df_add(g2, df_mul(q, d2));
}

// Convergence verdict on one evaluation: the double-float total of every
// CTA's per-warp partials (fixed order: rank, then warp), read through
// distributed shared memory.
template <class SH>
__device__ __forceinline__ Verdict residual_verdict(const SH &sh, const Part &pt, int buf, int64_t done,
                                         const df &thresh2, bool want_k, int64_t max_iter) {
    const int nw = (int)(blockDim.x >> 5), total = pt.C * nw, lane = threadIdx.x & 31;
    df r2 = df_from(0.f), k2 = df_from(0.f);
    for (int j = lane; j < total; j += 32) {
        const int r = j / nw, w = j - r * nw;
        r2 = df_add_f(r2, sh.ownp[r][(buf * 2 + 0) * kMaxWarps + w]);
        if (want_k) k2 = df_add_f(k2, sh.ownp[r][(buf * 2 + 1) * kMaxWarps + w]);
    }
    for (int o = 16; o > 0; o >>= 1) {
        r2 = df_add(r2, {__shfl_xor_sync(0xffffffffu, r2.hi, o), __shfl_xor_sync(0xffffffffu, r2.lo, o)});
        if (want_k)
            k2 = df_add(k2, {__shfl_xor_sync(0xffffffffu, k2.hi, o), __shfl_xor_sync(0xffffffffu, k2.lo, o)});
    }
    Verdict v;
    v.code = !isfinite(r2.hi) ? RVE_NAN : df_le(r2, thresh2) ? RVE_OK : done >= max_iter ? RVE_MAXITER : -1;
    v.r2h = r2.hi; v.r2l = r2.lo; v.k2h = k2.hi; v.k2l = k2.lo;
    return v;
}

// The residual test of the table kernels. Every thread leaves its squared
// residual (and kinetic energy); one warp per CTA adds them, FP32 within a warp
// and double-float over the warps, and sends the sum to every CTA; any warp can
// then total an evaluation and judge it.
constexpr int kRsStride = 36;  // floats per warp: 16-byte reads without bank conflicts
struct ResidualSums {
    float rs[2][kMaxWarps][kRsStride];  // by evaluation parity: the threads' squared residuals
    float ke[2][kMaxWarps][kRsStride];  // and kinetic energies
    float2 sum[3][2][kMaxParts];        // every CTA's (residual, kinetic) sums of three evaluations
};

// The sum of 32 floats in the order of an xor butterfly (16, 8, 4, 2, 1).
__device__ __forceinline__ float tree32(const float *v) {
    float b[16];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float4 x = *reinterpret_cast<const float4 *>(v + 4 * i), y = *reinterpret_cast<const float4 *>(v + 16 + 4 * i);
        b[4 * i] = x.x + y.x; b[4 * i + 1] = x.y + y.y; b[4 * i + 2] = x.z + y.z; b[4 * i + 3] = x.w + y.w;
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1)
#pragma unroll
        for (int i = 0; i < o; ++i) b[i] += b[i + o];
    return b[0];
}

// Double-float sum over each half-warp.
__device__ __forceinline__ df half_warp_sum(df t) {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1)
        t = df_add(t, {__shfl_xor_sync(0xffffffffu, t.hi, o), __shfl_xor_sync(0xffffffffu, t.lo, o)});
    return t;
}

// Testing warp: this CTA's sums of the evaluation with parity `q` (residual in
// the lower half-warp, kinetic energy in the upper) to entry `buf` of every CTA.
__device__ __forceinline__ void publish_sums(ResidualSums &sh, int q, int buf, int me, int C, bool want_k) {
    const int lane = threadIdx.x & 31, nw = (int)(blockDim.x >> 5), w = lane & 15, ke = lane >> 4;
    float v = 0.f;
    if (w < nw && (!ke || want_k)) v = tree32(ke ? sh.ke[q][w] : sh.rs[q][w]);
    const df t = half_warp_sum(df_from(v));
    if (w >= C || (ke && !want_k)) return;
    const uint32_t a = cluster_addr(smem_addr(&sh.sum[buf][ke][me]), (uint32_t)w);
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" :: "r"(a), "f"(t.hi), "f"(t.lo) : "memory");
}

// Convergence verdict on one evaluation from the CTAs' sums (every lane of the
// warp calls it and gets it).
__device__ __forceinline__ Verdict sums_verdict(const ResidualSums &sh, int buf, int C, df thresh2, int64_t done,
                                                bool want_k, int64_t max_iter) {
    const int lane = threadIdx.x & 31;
    df t = df_from(0.f);
    if ((lane & 15) < C && (lane < 16 || want_k)) {
        const float2 x = sh.sum[buf][lane >> 4][lane & 15];
        t = {x.x, x.y};
    }
    if (C > 1) t = half_warp_sum(t);
    Verdict v;
    v.r2h = __shfl_sync(0xffffffffu, t.hi, 0);
    v.r2l = __shfl_sync(0xffffffffu, t.lo, 0);
    v.k2h = __shfl_sync(0xffffffffu, t.hi, 16);
    v.k2l = __shfl_sync(0xffffffffu, t.lo, 16);
    v.code = !isfinite(v.r2h) ? RVE_NAN : df_le({v.r2h, v.r2l}, thresh2) ? RVE_OK : done >= max_iter ? RVE_MAXITER : -1;
    return v;
}

// End of a mixed solve of RVE p: the final displacement (FP64 output; the
// double-float displacement plus, with `add`, inc(k) of own free node k), the
// FP64 stress sum split across the cluster, and the per-RVE outputs.
template <class SH, class Inc>
__device__ __forceinline__ void mixed_finish(cg::cluster_group &cl, SH &sh, const DevMesh &M, const DevState &S,
                             const DevResults &O, const SolveParams &P, int p, const RveDesc &R,
                             const Part &pt, const double *F, bool add, const Inc &inc, int status, int64_t it,
                             df r2, df k2, double f_ref) {
    const int n = R.n_nodes, m = pt.m();
    const int64_t n0 = R.node0, b3 = 3 * n0;
    const float *uh = S.uh + b3, *ul = S.ul + b3;
    double *xg = S.xg + b3;
    const bool want_k = P.want_ke != 0;
    // ---- final displacement (FP64 output) and positions for the stress ----
    for (int k = threadIdx.x; k < m; k += blockDim.x) {
        const int i = pt.gidx(k);
        float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
        if (add && k < pt.nfr) d = inc(k);
        const float dd[3] = {d.x, d.y, d.z};
        double *uo[3] = {S.u0 + n0, S.u1 + n0, S.u2 + n0};
        const double *Xd[3] = {M.X0 + n0, M.X1 + n0, M.X2 + n0};
        for (int c = 0; c < 3; ++c) {
            df u = {uh[c * n + i], ul[c * n + i]};
            if (add && k < pt.nfr) u = df_add_f(u, dd[c]);
            const double ud = df_to_double(u);
            uo[c][i] = ud;
            xg[c * n + i] = dadd(Xd[c][i], ud);
        }
    }
    cl.sync();
    // stress: elements split across the cluster, partials reduced on rank 0
    double s[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) s[k] = 0.0;
    {
        const double *x0 = xg, *x1 = xg + n, *x2 = xg + 2 * n;
        for (int e = pt.me * blockDim.x + threadIdx.x; e < R.n_elems; e += pt.C * blockDim.x) {
            const int64_t ee = R.elem0 + e;
            const int a = M.el_a[ee], bb = M.el_b[ee];
            double d[3] = {dsub(x0[bb], x0[a]), dsub(x1[bb], x1[a]), dsub(x2[bb], x2[a])};
            const double l = dsqrt(dadd(dadd(dmul(d[0], d[0]), dmul(d[1], d[1])), dmul(d[2], d[2])));
            const double q = ddiv(dmul(M.el_EA[ee], dsub(ddiv(l, M.el_L[ee]), 1.0)), l);
#pragma unroll
            for (int rr = 0; rr < 3; ++rr)
#pragma unroll
                for (int c = 0; c < 3; ++c) s[3 * rr + c] = dadd(s[3 * rr + c], dmul(dmul(q, d[rr]), d[c]));
        }
    }
    {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            double v = s[k];
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) sh.wsum[warp][k] = v;
        }
    }
    __syncthreads();
    if (threadIdx.x < 9) {
        double t = 0.0;
        for (int w = 0; w < (int)((blockDim.x + 31) >> 5); ++w) t += sh.wsum[w][threadIdx.x];
        sh.sigp[pt.me * 9 + threadIdx.x] = t;
    }
    cl.sync();
    if (pt.me == 0 && threadIdx.x < 9) {
        double t = 0.0;
        for (int q = 0; q < pt.C; ++q) t += sh.sig[q][threadIdx.x];
        O.sigma[9 * (int64_t)p + threadIdx.x] = ddiv(t, dmul(det3(F), R.V0));
    }
    if (pt.me == 0 && threadIdx.x == 0) {
        const double r = sqrt(df_to_double(r2));
        O.iters[p] = it;
        O.rel_res[p] = f_ref > 0.0 ? r / f_ref : (r > 0.0 ? INFINITY : 0.0);
        O.status[p] = status;
        O.ke[p] = want_k ? df_to_double(k2) : 0.0;
    }
    cl.sync();
}

// The next iteration's partial velocity update (Algorithm 1: v += dt/2 a)
// and displacement increment (u += dt v, as an increment on top of d) for one
// node, from its velocity w and acceleration a after this iteration.
__device__ __forceinline__ void next_increment(float w0, float w1, float w2, float a0, float a1, float a2,
                                               const float4 &d, float hdtf, float dtf, float4 &sv,
                                               float2 &sa, float4 &next) {
    const float v0 = w0 + hdtf * a0, v1 = w1 + hdtf * a1, v2 = w2 + hdtf * a2;
    sv = make_float4(v0, v1, v2, a0);
    sa = make_float2(a1, a2);
    next = make_float4(d.x + dtf * v0, d.y + dtf * v1, d.z + dtf * v2, 0.f);
}


}  // namespace
}  // namespace fe2
