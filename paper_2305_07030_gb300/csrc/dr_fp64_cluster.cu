// FP64 dynamic relaxation (Algorithm 1) of one RVE on a thread-block cluster.
//
// Each RVE is split into parts, one per CTA of a cluster of 1 to 16 CTAs. The
// paper used one team per sub-problem (Section III); a cluster is a team that
// spans SMs.
//
// Arithmetic is that of a serial element-scatter implementation, operation for
// operation, so the trajectory is the oracle's bit for bit:
//  * each CTA keeps its own nodes' positions in shared memory (two buffers,
//    one per evaluation parity) and reads neighbours of other parts through
//    distributed shared memory;
//  * each element with an end among the CTA's free nodes has a slot in the
//    CTA's element table; its force on the first end is evaluated once per
//    iteration;
//  * each free node sums the +- slot forces of its row in row order, then the
//    damping, acceleration and velocity updates follow. The next iteration's
//    partial velocity update and displacement come right after them, from
//    the same product dt/2 a, so the acceleration is never stored.
//
// Synchronisation. One cluster barrier per iteration, before the element
// forces, and one CTA barrier after them. The residual test runs beside the
// element forces: at evaluation i the terms of evaluation i-1 are summed by a few
// warps of each CTA, and one judging warp per CTA, which evaluates no elements,
// totals evaluation i-2 across the cluster (a tree, the same bits in every CTA).
// The workers read its verdict after the CTA barrier. The displacements
// of the last three evaluations rotate through a ring in global memory (L2),
// so the tested evaluation's state is still there.
//
// Sums. Every sum over the nodes goes leaf by leaf (Leaves below), so an RVE's
// results do not depend on how many CTAs its batch leaves for it. The chains of
// dependent additions are what a test costs: under load an FP64 instruction of a
// warp waits for the pipe for 100 to 250 cycles. A leaf's terms are therefore spread
// over groups of about 64 nodes and 32 lanes each, one group to a warp, and warps
// without elements do it first; kinetic energies are kept for three evaluations and
// summed at the end. Per iteration, with sums by thread, warp and CTA in the judging
// warp alone (which the batch could change) and so: 512 nodes on 8 CTAs 4.3 -> 3.8 us
// (energy check 8.4 -> 5.3), 152 RVEs of 200 nodes 6.45 -> 6.35 (10.5 -> 8.1), of 800 17.9 ->
// 17.5 (23.8 -> 25.3), 5000 nodes on 16 CTAs 9.85 -> 9.2 (14.6 -> 12.6), 60,000 90.3 -> 86.7
// (117 -> 123). The energy check costs up to 6 % more than it did where its terms are
// many (parts of 800 nodes and more). Two groups to a warp: 200 nodes 6.85, 5000 9.6 us;
// four: 7.6, 10.2; with one judging lane per 32 / leaves of a CTA 512 nodes 6.1.
//
// What bounds it: the FP64 pipe, 2 operations per clock and SM. Per element 13
// additions and multiplications, per free node 45 at degree 5; divisions and
// square roots run on the integer pipes (f64_soft.cuh). Everything that is the
// same for the whole CTA is kept off that pipe: a residual total or a square
// root computed by every thread costs 16 warps' slots. Measured per
// iteration, before (totals in every thread, the acceleration stored, the
// update a phase of its own, one-part RVEs on the single-CTA kernel) and now:
// 5000 nodes on 8 CTAs 23.4 -> 15.8 us, 512 nodes on one CTA 18.8 -> 12.2 us.
#include <cooperative_groups.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <utility>

#include "dr_device.cuh"

namespace cg = cooperative_groups;

namespace fe2 {

namespace {

// Threads per CTA at most; the last warp judges. 16 warps are 4 per scheduler
// and leave 128 registers per thread (17 would leave 96, and spills).
constexpr int kMaxThreads = 512;
constexpr int kRegElems = 3;      // table elements a worker keeps in registers

struct Fp64ClusterShared {
    double part[2][4][kMaxParts];    // sums of this CTA's groups for evaluation n (parity n & 1):
                                     // squared residual, kinetic energy, work terms
    const double *partp[kMaxParts];  // every CTA's `part`
    double sig[kStressWarps][9];     // stress partials (rank 0's copy is the target)
    double *sigp;                    // rank 0's sig
    int code;                        // verdict: -1 = go on, else the RVE status
    int item;
};

__device__ __forceinline__ void cl_arrive() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void cl_wait() {
    asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

// The leaves of an RVE (fe2_internal.h): its sums are formed leaf by leaf, each
// in an order of its own, so they are the same bits whatever the cluster size,
// the CTA size and the other RVEs of the batch.
struct Leaves {
    const uint16_t *list;  // this CTA's nodes by leaf; null: one leaf, in order
    const int32_t *off;    // first entries of this CTA's leaves, counted from the RVE's
    const int32_t *free;   // their free nodes
    int own, total;        // leaves of this CTA and of the RVE (powers of two)
    int base;              // the CTA's first entry
};
__device__ __forceinline__ Leaves make_leaves(const DevMesh &M, const RveDesc &R, int p, int me, int C, int c0) {
    Leaves l;
    l.total = R.fp_leaves;
    l.own = l.total / C;
    l.base = c0;
    l.list = l.own > 1 ? M.fp_leaf + R.node0 + c0 : nullptr;
    l.off = M.fp_leaf_off + (int64_t)p * 2 * (kMaxParts + 1) + me * l.own;
    l.free = l.off + (kMaxParts + 1);
    return l;
}

// Sum over the RVE of one value per own node (set-up only; `parity` picks the
// publication buffer). Every thread gets the total; a cluster barrier.
__device__ __forceinline__ double node_sum(cg::cluster_group &cl, Fp64ClusterShared &sh, const Leaves &lv,
                                           const double *v, int m, int parity) {
    const int lane = threadIdx.x & 31;
    __syncthreads();
    for (int j = threadIdx.x >> 5; j < lv.own; j += blockDim.x >> 5) {
        const int beg = lv.list ? lv.off[j] - lv.base : 0, end = lv.list ? lv.off[j + 1] - lv.base : m;
        double t = 0.0;
        for (int q = beg + lane; q < end; q += 32) t = dadd(t, v[lv.list ? lv.list[q] : q]);
        for (int o = 16; o > 0; o >>= 1) t = dadd(t, __shfl_xor_sync(0xffffffffu, t, o));
        if (lane == 0) sh.part[parity][0][j] = t;
    }
    cl.sync();
    double s = 0.0;
    for (int l = 0; l < lv.total; ++l)
        s = dadd(s, sh.partp[l / lv.own][parity * 4 * kMaxParts + l % lv.own]);
    return s;
}

// Position component at a shared-memory address: shared::cta, or
// shared::cluster with bit 0 set for another CTA's node.
__device__ __forceinline__ double ld_pos(uint32_t a) {
    double v;
    if (a & 1u) asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a & ~1u));
    else asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(a));
    return v;
}

// One table element: rigidity, reference length and its division estimate,
// the two ends' positions in buffer 0.
struct Slot {
    double EA, L;
    uint32_t vL, a, b;
};

__device__ __forceinline__ uint32_t pos_addr(const double *XB, int ref, int me) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(XB + (ref & 0xffff));
    const int r = ref >> 16;
    if (r == me) return a;
    uint32_t c;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(c) : "r"(a), "r"(r));
    return c | 1u;
}

__device__ __forceinline__ Slot load_slot(const DevMesh &M, const RveDesc &R, const int4 *slots, int s,
                                          const double *XB, int me) {
    const int4 sl = slots[s];
    Slot e;
    e.EA = M.el_EA[R.elem0 + sl.x];
    e.L = M.el_L[R.elem0 + sl.x];
    e.vL = f64_recip_of(e.L);
    e.a = pos_addr(XB, sl.y, me);
    e.b = pos_addr(XB, sl.z, me);
    return e;
}

// Force on the element's first end, t = (N/l) d, into T[0], T[ts], T[2 ts].
// boff: the position buffer's byte offset, cb: a component's.
__device__ __forceinline__ void slot_force(const Slot &e, uint32_t boff, uint32_t cb, double *T, int ts) {
    const uint32_t a = e.a + boff, b = e.b + boff;
    const double a0 = ld_pos(a), a1 = ld_pos(a + cb), a2 = ld_pos(a + 2 * cb);
    const double b0 = ld_pos(b), b1 = ld_pos(b + cb), b2 = ld_pos(b + 2 * cb);
    const double d0 = dsub(b0, a0), d1 = dsub(b1, a1), d2 = dsub(b2, a2);
    uint32_t vl;
    const double l = f64_sqrt_recip(dadd(dadd(dmul(d0, d0), dmul(d1, d1)), dmul(d2, d2)), vl);
    const double N = dmul(e.EA, dsub(f64_div_v<false>(l, e.L, e.vL), 1.0));
    const double q = f64_div_v<true>(N, l, vl);
    T[0] = dmul(q, d0);
    T[ts] = dmul(q, d1);
    T[2 * ts] = dmul(q, d2);
}

// Doubles per free node of the state in shared memory, by Fp64Shape::ssm: velocity,
// reference position, mass, damping factor, the mass's division estimate, the
// force's squares; displacement unless 2.
__host__ __device__ constexpr size_t state_doubles(int ssm) { return ssm == 1 ? 15 : ssm == 2 ? 12 : 0; }

// Doubles per free node of the energy terms in shared memory.
__host__ __device__ constexpr size_t term_doubles(bool terms) { return terms ? 9 : 0; }

// Dynamic shared memory of a launch shape (layout: cluster_tables).
__host__ __device__ inline size_t cluster_bytes(const Fp64Shape &sp) {
    size_t b = sizeof(double) * (6 * (size_t)sp.part_max + (state_doubles(sp.ssm) + term_doubles(sp.terms)) * (size_t)sp.free_max);
    if (sp.tsm)
        b += sizeof(double) * 3 * (size_t)sp.slot_max + sizeof(int32_t) * ((size_t)sp.free_max + 1) +
             sizeof(uint16_t) * (size_t)sp.row_max;
    if (sp.ssm == 1) b += sizeof(uint16_t) * (size_t)sp.part_max;
    return (b + 15) & ~size_t(15);
}

}  // namespace

// One RVE on the cluster. XB (smem) is this CTA's [2][3][part_cap] position
// buffers. With TSM the element table T [3][slot_cap] and the rows (RS: first
// entry of each free node, RE: entries slot << 1 | second end) are in shared
// memory, otherwise in global memory. With SSM = 1 the own free nodes' state (ST:
// velocity, reference position, the force's squares [3][free_cap] each, mass,
// damping factor -c m and the mass's division estimate [free_cap] each, displacement
// [3][free_cap]) and the list of the nodes by leaf (LS) are in shared memory, with
// SSM = 2 all but the displacement (from the ring) and the list, otherwise in global
// memory (L2). 2 is for parts that 1 does not fit. TE: the kinetic energies of three
// evaluations, or one's with the two work terms (energy check), of the free nodes,
// [3][free_cap] each, null for global memory.
template <bool TSM, int SSM>
__device__ void solve_rve_fp64_cluster(cg::cluster_group &cl, Fp64ClusterShared &sh, const DevMesh &M,
                                       const DevState &S, const DevResults &O, const SolveParams &P, int p,
                                       double *XB, double *ST, double *TE, double *Tsm, int32_t *RS, uint16_t *RE, uint16_t *LS,
                                       int part_cap, int free_cap, int slot_cap) {
    const RveDesc R = M.rve[p];
    const int me = (int)cl.block_rank(), C = (int)cl.num_blocks();
    const int W = blockDim.x - 32;  // workers; the last warp judges
    const int tid = threadIdx.x, lane = tid & 31;
    const bool judge = tid >= W;
    const int32_t *po = M.fp_part_off + (int64_t)p * 2 * (kMaxParts + 1);
    const int n = R.n_nodes;
    const int c0 = po[me], m = po[me + 1] - c0;  // own nodes: positions c0 .. of the FP64 order
    const int f0 = po[kMaxParts + 1 + me], nfr = po[kMaxParts + 1 + me + 1] - f0;  // own free nodes
    const int64_t n0 = R.node0;
    const int32_t *node = M.fp_node + n0 + c0;      // their RVE-local ids, free nodes first
    const int32_t *rowptr = M.rowptr + R.rp0;
    const int32_t *frow = M.fp_row + R.rp0 + f0;
    const int32_t *fent = M.fp_csr_slot + R.csr0;
    const int32_t *ps = M.fp_part_slot + (int64_t)p * (kMaxParts + 1);
    const int s0 = ps[me], ns = ps[me + 1] - s0;
    const int4 *slots = M.fp_slot + R.slot0 + s0;
    const int ts = TSM ? slot_cap : ns;
    double *T = TSM ? Tsm : S.fpt + 3 * (R.slot0 + s0);
    double F[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) F[k] = P.F[9 * (int64_t)p + k];
    const double *X0 = M.X0 + n0, *X1 = M.X1 + n0, *X2 = M.X2 + n0;
    double *xg = S.xg + 3 * n0;
    // displacements of the free nodes by FP64 order, evaluation i in ring i % 3
    double *const ring = S.ualt + 9 * n0 + c0;
    const int rstride = 3 * n;
    const uint32_t cb = (uint32_t)(sizeof(double) * part_cap);
    const bool energy = P.want_ke == 2;
    double *gp = S.gp + 3 * n0 + c0, *fdp = S.fdp + 3 * n0 + c0;  // by FP64 order, energy check
    double *const sv = ST, *const sx = ST + 3 * free_cap, *const su = ST + 12 * free_cap;
    double *const sm = ST + 9 * free_cap, *const sc = ST + 10 * free_cap;
    uint32_t *const sr = reinterpret_cast<uint32_t *>(ST + 11 * free_cap);
    double *const gv = S.v0 + n0 + c0;  // !SSM: component c at c * vstride
    const int64_t vstride = S.v1 - S.v0;
    const double mc = -R.c;
    // squares of the free nodes' forces; kinetic energies and work terms
    double *const G2 = SSM ? ST + 6 * free_cap : xg + c0;
    const int gs = SSM ? free_cap : n;
    // Without the energy check the kinetic energies are wanted at the end only: those of
    // the last three evaluations are kept (slot by displacement ring index).
    const bool ke_ring = P.want_ke == 1;
    const int64_t gstride = S.a1 - S.a0, kstride = TE ? free_cap : gstride;
    double *const kt = TE ? TE : S.a0 + n0 + c0;
    double *const wt = TE ? TE + 3 * free_cap : S.a0 + 3 * gstride + 6 * n0 + c0;
    const int wts = TE ? free_cap : n;
    auto ke_slot = [&](int slot) { return slot == 0 ? kt : wt + 3 * (slot - 1) * wts; };
    auto ke_stride = [&](int slot) { return slot == 0 ? kstride : (int64_t)wts; };
    const Leaves lv = make_leaves(M, R, p, me, C, c0);
    double *const nn = ring + 2 * rstride;  // set-up: one value per own node

    // f_ref, part 1: forces in the affine configuration x = F X (all DOFs)
    for (int k = tid; k < m; k += blockDim.x) {
        const int i = node[k];
        const double Xv[3] = {X0[i], X1[i], X2[i]};
        for (int r = 0; r < 3; ++r)
            xg[r * n + i] = dadd(dadd(dmul(F[3 * r], Xv[0]), dmul(F[3 * r + 1], Xv[1])), dmul(F[3 * r + 2], Xv[2]));
    }
    cl.sync();
    for (int k = tid; k < m; k += blockDim.x) {
        double g0, g1, g2;
        gather_force_fp64(M, rowptr, R.csr0, node[k], xg, xg + n, xg + 2 * n, g0, g1, g2);
        nn[k] = dadd(dadd(dmul(g0, g0), dmul(g1, g1)), dmul(g2, g2));
    }
    const double f_aff = dsqrt(node_sum(cl, sh, lv, nn, m, 0));

    // Algorithm 1: displacement BCs on fixed nodes, initial free displacement
    for (int k = tid; k < m; k += blockDim.x) {
        const int i = node[k];
        const bool fixed = k >= nfr;
        const double Xv[3] = {X0[i], X1[i], X2[i]};
        double *const uo[3] = {S.u0 + n0, S.u1 + n0, S.u2 + n0};
        for (int r = 0; r < 3; ++r) {
            const double uaff = dsub(xg[r * n + i], Xv[r]);
            const double u = fixed || P.init == 1 ? uaff : (P.init == 2 ? uo[r][i] : 0.0);
            const double x = dadd(Xv[r], u);
            uo[r][i] = u;
            xg[r * n + i] = x;
            XB[r * part_cap + k] = x;
            XB[(3 + r) * part_cap + k] = x;  // fixed positions live in both buffers
            if (SSM && !fixed) {
                if (SSM == 1) su[r * free_cap + k] = u;
                sx[r * free_cap + k] = Xv[r];
            }
            if (!fixed) ring[r * n + k] = u;
        }
        if (SSM && !fixed) {
            const double mm = M.mass[n0 + i];
            sm[k] = mm;
            sc[k] = dmul(mc, mm);
            sr[k] = f64_recip_of(mm);
        }
    }
    if (TSM) {
        for (int k = tid; k <= nfr; k += blockDim.x) RS[k] = frow[k] - frow[0];
        const int ne = frow[nfr] - frow[0];
        for (int q = tid; q < ne; q += blockDim.x) RE[q] = (uint16_t)fent[frow[0] + q];
    }
    if (SSM == 1 && lv.list)
        for (int k = tid; k < m; k += blockDim.x) LS[k] = lv.list[k];
    Slot el[kRegElems];
#pragma unroll
    for (int j = 0; j < kRegElems; ++j) {
        el[j] = Slot{};
        if (!judge && tid + j * W < ns) el[j] = load_slot(M, R, slots, tid + j * W, XB, me);
    }
    if (tid == 0) sh.code = -1;
    cl.sync();
    const double dt = dmul(P.alpha, R.dtc);  // compute next time step (constant)
    const double hdt = dmul(0.5, dt);
    // getInternalForces(u); accelerations; the first partial velocity update
    // and displacement (free DOFs)
    for (int k = tid; k < m; k += blockDim.x) {
        const int i = node[k];
        double g[3];
        gather_force_fp64(M, rowptr, R.csr0, i, xg, xg + n, xg + 2 * n, g[0], g[1], g[2]);
        nn[k] = dadd(dadd(dmul(g[0], g[0]), dmul(g[1], g[1])), dmul(g[2], g[2]));
        if (k < nfr) {
            const double mm = M.mass[n0 + i];
            const double Xv[3] = {X0[i], X1[i], X2[i]};
            for (int r = 0; r < 3; ++r) {
                const double v = dadd(0.0, dmul(hdt, ddiv(g[r], mm)));
                const double u = dadd(ring[r * n + k], dmul(dt, v));
                ring[rstride + r * n + k] = u;
                XB[(3 + r) * part_cap + k] = dadd(Xv[r], u);
                if (SSM) {
                    sv[r * free_cap + k] = v;
                    if (SSM == 1) su[r * free_cap + k] = u;
                } else {
                    gv[r * vstride + k] = v;
                }
                if (energy) {
                    // the work sums start from the initial force and no damping force
                    gp[r * n + k] = g[r];
                    fdp[r * n + k] = 0.0;
                }
            }
        }
    }
    const double f0v = dsqrt(node_sum(cl, sh, lv, nn, m, 1));
    const double f_ref = f_aff > f0v ? f_aff : f0v;
    const double thresh = P.tol * f_ref;
    double res = 0.0, ke = 0.0, wint = 0.0, wext = 0.0;  // judging warp: of the last tested evaluation
    int rc = 1;                                          // ring index of evaluation i
    // Sums of the terms of evaluation i - 1, for every kind of term and every group of
    // a leaf's terms: entry y = 3 j + c (component c of the leaf's free node j) belongs
    // to lane y mod 32 of group (y / 32) mod groups, and the lanes' sums are added as a
    // tree. A warp takes one kind and one group at a time, two where there are more
    // than warps; the last warps, which have the fewest elements, begin, and the judging
    // warp comes last where others have none.
    const int gsh = 31 - __clz(R.fp_groups), ush = 31 - __clz(lv.own) + gsh;  // 2^ush groups here
    const int kinds = energy ? 4 : 1;
    const int nw = (int)(blockDim.x >> 5), from_end = nw - 1 - (tid >> 5);
    const int first_sum = ns > W - 32 ? from_end : from_end == 0 ? nw - 1 : from_end - 1;
    const int all_groups = lv.total << gsh;
    auto pair_of = [&](int kinds_now) { return ush > 0 && kinds_now << ush > nw ? 1 : 0; };
    const int pair = pair_of(kinds);
    const double *const lsum =  // the group's sums that this lane adds first
        lane < all_groups ? sh.partp[lane >> ush] + (lane & ((1 << ush) - 1)) : nullptr;
    auto lane_sum = [&](const double *v, int64_t vs, int u) {
        const int l = u >> gsh, beg = lv.list ? lv.off[l] - lv.base : 0;
        const int end = 3 * (lv.list ? lv.free[l] : nfr);
        auto term = [&](int y) {
            const int j = beg + y / 3, k = lv.list ? (SSM == 1 ? LS[j] : lv.list[j]) : j;
            return v[(y % 3) * vs + k];
        };
        int y = lane + 32 * (u & ((1 << gsh) - 1));
        double t = y < end ? term(y) : 0.0;
#pragma unroll 4
        for (y += 32 << gsh; y < end; y += 32 << gsh) t = dadd(t, term(y));
        return t;
    };
    // terms `v` ([3] components `vs` apart) of group u (and u + 1 with `two`) into out
    auto group_sums = [&](const double *v, int64_t vs, int u, int two, double *out) {
        double t = lane_sum(v, vs, u), o = t;
        if (two) {  // lanes 0 to 15 go on with the first group, 16 to 31 with the second
            const double t2 = lane_sum(v, vs, u + 1);
            o = (lane & 16) ? t : t2;
            t = (lane & 16) ? t2 : t;
        }
        t = dadd(t, __shfl_xor_sync(0xffffffffu, o, 16));
        for (int d = 8; d > 0; d >>= 1) t = dadd(t, __shfl_xor_sync(0xffffffffu, t, d));
        if ((lane & 15) == 0 && (lane == 0 || two)) out[u + (lane >> 4)] = t;
    };
    auto leaf_sums = [&](int64_t ev) {
        for (int x = first_sum; x < kinds << (ush - pair); x += nw) {
            const int kind = x >> (ush - pair), u = (x & ((1 << (ush - pair)) - 1)) << pair;
            const double *const v = kind == 0 ? G2 : kind == 1 ? kt : kind == 2 ? wt : wt + 3 * wts;
            group_sums(v, kind == 0 ? gs : kind == 1 ? kstride : wts, u, pair, sh.part[ev & 1][kind]);
        }
    };
    // the RVE's total of one kind, from the groups' sums of parity q: a tree over the
    // lanes, the same bits in every CTA
    auto total = [&](int kind, int q) {
        const int at = (q * 4 + kind) * kMaxParts;
        double t = lsum ? lsum[at] : 0.0;
        for (int e = lane + 32; e < all_groups; e += 32)
            t = dadd(t, sh.partp[e >> ush][at + (e & ((1 << ush) - 1))]);
        for (int o = 1; o < 32 && o < all_groups; o <<= 1) t = dadd(t, __shfl_xor_sync(0xffffffffu, t, o));
        return t;
    };
    int64_t i = 1;
    for (;; ++i) {
        const uint32_t boff = (i & 1) ? 3 * cb : 0u;
        // positions of evaluation i, and the CTA sums of evaluation i-2,
        // become visible to the whole cluster
        if (C > 1) {
            cl_arrive();
            cl_wait();
        } else {
            __syncthreads();
        }
        if (!judge) {
#pragma unroll
            for (int j = 0; j < kRegElems; ++j)
                if (tid + j * W < ns) slot_force(el[j], boff, cb, T + tid + j * W, ts);
            for (int s = tid + kRegElems * W; s < ns; s += W)
                slot_force(load_slot(M, R, slots, s, XB, me), boff, cb, T + s, ts);
            if (i >= 2) leaf_sums(i - 1);
        } else {
            if (i >= 2) leaf_sums(i - 1);
            if (i >= 3) {  // verdict on evaluation i-2
                const int q = (int)(i & 1);
                res = dsqrt(total(0, q));
                if (energy) {
                    ke = total(1, q);
                    wint = dsub(wint, dmul(0.5, total(2, q)));
                    wext = dadd(wext, dmul(0.5, total(3, q)));
                }
                const int code = !isfinite(res) ? RVE_NAN : res <= thresh ? RVE_OK : i - 2 >= P.max_iter ? RVE_MAXITER : -1;
                if (lane == 0) sh.code = code;
            }
        }
        __syncthreads();
        if (sh.code >= 0) break;
        // getInternalForces (slot sums in row order); damping force; residual;
        // accelerations; velocity; the next partial velocity update and
        // displacement. One item per free DOF (component-major), which evens
        // the work out over the warps.
        const int rn = rc == 2 ? 0 : rc + 1;
        if (!judge) {
            double *const xn = XB + ((i & 1) ? 0 : 3 * part_cap);
            const double *const up = ring + rc * rstride;
            double *const un = ring + rn * rstride;
            double *const kn = ke_slot(ke_ring ? rc : 0);
            const int64_t kns = ke_stride(ke_ring ? rc : 0);
            for (int x = tid; x < 3 * nfr; x += W) {
                const int c = (x >= nfr) + (x >= 2 * nfr), k = x - c * nfr;
                const double *Tc = T + c * ts;
                double g = 0.0;
                int q = TSM ? RS[k] : frow[k];
                const int end = TSM ? RS[k + 1] : frow[k + 1];
                for (; q < end; ++q) {
                    const uint32_t w = TSM ? (uint32_t)RE[q] : (uint32_t)fent[q];
                    // the second end receives -t
                    g = dadd(g, f64_from(f64_bits(Tc[w >> 1]) ^ ((uint64_t)(w & 1u) << 63)));
                }
                double mm, cm, vv, uu, xr;
                uint32_t vm;
                if (SSM) {
                    mm = sm[k]; cm = sc[k]; vm = sr[k];
                    vv = sv[c * free_cap + k]; uu = SSM == 1 ? su[c * free_cap + k] : up[c * n + k]; xr = sx[c * free_cap + k];
                } else {
                    const int id = node[k];
                    mm = M.mass[n0 + id];
                    cm = dmul(mc, mm);
                    vm = f64_recip_of(mm);
                    vv = gv[c * vstride + k]; uu = up[c * n + k]; xr = c == 0 ? X0[id] : (c == 1 ? X1[id] : X2[id]);
                }
                const double fd = dmul(cm, vv);
                G2[c * gs + k] = dmul(g, g);
                if (energy) {
                    const double du = dmul(dt, vv);
                    wt[c * wts + k] = dmul(du, dadd(gp[c * n + k], g));
                    wt[(3 + c) * wts + k] = dmul(du, dadd(fdp[c * n + k], fd));
                    gp[c * n + k] = g;
                    fdp[c * n + k] = fd;
                }
                const double ha = dmul(hdt, f64_div_v<false>(dadd(g, fd), mm, vm));
                const double v1 = dadd(vv, ha);
                if (P.want_ke) kn[c * kns + k] = dmul(dmul(0.5, mm), dmul(v1, v1));
                const double vh = dadd(v1, ha);
                const double u = dadd(uu, dmul(dt, vh));
                if (SSM) {
                    sv[c * free_cap + k] = vh;
                    if (SSM == 1) su[c * free_cap + k] = u;
                } else {
                    gv[c * vstride + k] = vh;
                }
                un[c * n + k] = u;
                xn[c * part_cap + k] = dadd(xr, u);
            }
        }
        rc = rn;
    }
    // The stopping evaluation is i - 2, ring index (i - 2) % 3 = (i + 1) % 3:
    // final displacement to the output arrays, positions to the global scratch
    const int rf = rc == 2 ? 0 : rc + 1;
    const double *const uf = ring + rf * rstride;
    if (ke_ring) {
        const int two = pair_of(1);
        for (int x = tid >> 5; x < 1 << (ush - two); x += nw)
            group_sums(ke_slot(rf), ke_stride(rf), x << two, two, sh.part[0][1]);
    }
    for (int k = tid; k < m; k += blockDim.x) {
        const int id = node[k];
        double *const uo[3] = {S.u0 + n0, S.u1 + n0, S.u2 + n0};
        const double Xv[3] = {X0[id], X1[id], X2[id]};
        for (int r = 0; r < 3; ++r) {
            if (k < nfr) uo[r][id] = uf[r * n + k];
            xg[r * n + id] = dadd(Xv[r], uo[r][id]);
        }
    }
    cl.sync();
    stress_partials(M, R, xg, xg + n, xg + 2 * n, me, C, sh.sigp);
    cl.sync();
    if (me == 0) {
        stress_total(R, F, &sh.sig[0][0], O.sigma + 9 * (int64_t)p);
        if (judge && ke_ring) ke = total(1, 0);
        if (judge && lane == 0) {
            O.iters[p] = i - 2;
            O.rel_res[p] = f_ref > 0.0 ? res / f_ref : (res > 0.0 ? INFINITY : 0.0);
            O.status[p] = sh.code;
            O.f_ref[p] = f_ref;
            O.ke[p] = ke;
            if (O.wint) O.wint[p] = wint;
            if (O.wext) O.wext[p] = wext;
        }
    }
    cl.sync();  // the next RVE may overwrite the buffers
}

namespace {
__device__ __forceinline__ void map_shared(cg::cluster_group &cl, Fp64ClusterShared &sh) {
    if ((int)threadIdx.x < (int)cl.num_blocks()) {
        const int r = threadIdx.x;
        sh.partp[r] = cl.map_shared_rank(&sh.part[0][0][0], r);
    }
    if (threadIdx.x == 0) sh.sigp = cl.map_shared_rank(&sh.sig[0][0], 0);
}

// One RVE with the tables of a launch shape in `base` (cluster_bytes).
template <bool TSM, int SSM>
__device__ __forceinline__ void solve_in(cg::cluster_group &cl, Fp64ClusterShared &sh, const DevMesh &M,
                                         const DevState &S, const DevResults &O, const SolveParams &P, int p,
                                         const Fp64Shape &sp, double *base) {
    double *XB = base;
    double *ST = XB + 6 * sp.part_max;
    double *TE = ST + state_doubles(SSM) * (size_t)sp.free_max;
    double *T = TE + term_doubles(sp.terms) * (size_t)sp.free_max;
    int32_t *RS = reinterpret_cast<int32_t *>(T + (TSM ? 3 * (size_t)sp.slot_max : 0));
    uint16_t *RE = reinterpret_cast<uint16_t *>(RS + (TSM ? sp.free_max + 1 : 0));
    uint16_t *LS = RE + (TSM ? sp.row_max : 0);
    solve_rve_fp64_cluster<TSM, SSM>(cl, sh, M, S, O, P, p, XB, ST, sp.terms ? TE : nullptr, T, RS, RE, LS, sp.part_max,
                                     sp.free_max, sp.slot_max);
}
}  // namespace

template <bool TSM, int SSM>
__global__ void __launch_bounds__(kMaxThreads, 1)
    dr_fp64_cluster_kernel(DevMesh M, DevState S, DevResults O, SolveParams P, Fp64Shape sp) {
    extern __shared__ __align__(16) double dsm_fp64[];
    __shared__ Fp64ClusterShared sh;
    cg::cluster_group cl = cg::this_cluster();
    map_shared(cl, sh);
    for (;;) {
        if (cl.block_rank() == 0 && threadIdx.x == 0) sh.item = atomicAdd(P.counter, 1);
        cl.sync();
        const int item = *cl.map_shared_rank(&sh.item, 0);
        cl.sync();
        if (item >= P.queue_len) return;
        solve_in<TSM, SSM>(cl, sh, M, S, O, P, P.queue[item], sp, dsm_fp64);
    }
}

// The allocation-free call: RVE 0, whose tables a packing kernel left in M's
// arrays, with the shared-memory variant its own capacities allow in `bytes`; the
// displacement goes to u in the caller's order (perm). Nothing is done when the
// packing kernel found the inputs invalid (*skip).
__global__ void __launch_bounds__(kMaxThreads, 1)
    dr_fp64_single_kernel(DevMesh M, DevState S, DevResults O, SolveParams P, size_t bytes, const int *skip,
                          const int32_t *perm, double *u) {
    extern __shared__ __align__(16) double dsm_fp64[];
    __shared__ Fp64ClusterShared sh;
    if (*skip) return;
    cg::cluster_group cl = cg::this_cluster();
    map_shared(cl, sh);
    cl.sync();
    const RveDesc &R = M.rve[0];
    Fp64Shape sp = {R.fp_parts, R.fp_part_max, R.fp_free_max, R.fp_slot_max, R.fp_row_max, true, 1, false};
    if (cluster_bytes(sp) <= bytes) {
        solve_in<true, 1>(cl, sh, M, S, O, P, 0, sp, dsm_fp64);
    } else {
        sp.tsm = false;
        sp.ssm = 0;
        solve_in<false, 0>(cl, sh, M, S, O, P, 0, sp, dsm_fp64);
    }
    const double *uo[3] = {S.u0, S.u1, S.u2};
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < R.n_nodes; k += gridDim.x * blockDim.x)
        for (int c = 0; c < 3; ++c) u[3 * perm[k] + c] = uo[c][k];
}

namespace {
using Fp64ClusterKernel = void (*)(DevMesh, DevState, DevResults, SolveParams, Fp64Shape);

Fp64ClusterKernel pick_fp64_cluster(const Fp64Shape &sp) {
    if (sp.tsm)
        return sp.ssm == 1 ? dr_fp64_cluster_kernel<true, 1>
                           : sp.ssm ? dr_fp64_cluster_kernel<true, 2> : dr_fp64_cluster_kernel<true, 0>;
    return sp.ssm == 1 ? dr_fp64_cluster_kernel<false, 1>
                       : sp.ssm ? dr_fp64_cluster_kernel<false, 2> : dr_fp64_cluster_kernel<false, 0>;
}

cudaLaunchConfig_t fp64_cluster_config(int clusters, const Fp64Shape &sp, int block, cudaLaunchAttribute *attr,
                                       cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(clusters * sp.parts, 1, 1);
    cfg.blockDim = dim3(block, 1, 1);
    cfg.dynamicSmemBytes = fp64_cluster_smem(sp);
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = sp.parts;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

// Raise the kernel's dynamic shared-memory limit (and allow 16-CTA
// clusters) once per device and size, so that launches recorded into a CUDA
// graph make no attribute calls of their own.
std::mutex g_fp64c_mutex;
std::map<std::pair<const void *, int>, int> g_fp64c_bytes;

void prepare_fp64_cluster(Fp64ClusterKernel k, size_t smem) {
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lock(g_fp64c_mutex);
    int &have = g_fp64c_bytes[{reinterpret_cast<const void *>(k), dev}];
    if (have == 0 || have < (int)smem) {
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        have = std::max(have, (int)smem);
    }
}
}  // namespace

size_t fp64_cluster_smem(const Fp64Shape &sp) { return cluster_bytes(sp); }

int launch_dr_fp64_cluster(const DevMesh &m, const DevState &s, const DevResults &r, const SolveParams &p,
                           int clusters, int block, const Fp64Shape &sp, void *stream) {
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = fp64_cluster_config(clusters, sp, block, attr, static_cast<cudaStream_t>(stream));
    const Fp64ClusterKernel k = pick_fp64_cluster(sp);
    prepare_fp64_cluster(k, cfg.dynamicSmemBytes);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k, m, s, r, p, sp);
    if (e != cudaSuccess) return (int)e;
    return (int)cudaGetLastError();
}

int occupancy_dr_fp64_cluster(int block, const Fp64Shape &sp) {
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = fp64_cluster_config(64, sp, block, attr, nullptr);
    const Fp64ClusterKernel k = pick_fp64_cluster(sp);
    prepare_fp64_cluster(k, cfg.dynamicSmemBytes);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

// Largest power of two up to kMaxParts of CTAs with `smem` bytes each that fit on
// the device as one cluster (0: not even one CTA).
template <class K>
static int largest_cluster(K kernel, size_t smem) {
    for (int c = kMaxParts; c > 0; c /= 2) {
        cudaLaunchAttribute attr[1];
        Fp64Shape sp = {};
        sp.parts = c;
        cudaLaunchConfig_t cfg = fp64_cluster_config(1, sp, kMaxThreads, attr, nullptr);
        cfg.dynamicSmemBytes = smem;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess && n > 0) return c;
        cudaGetLastError();
    }
    return 0;
}

// The same for the cluster kernel, once per device and size.
int fp64_max_cluster(size_t smem) {
    static std::mutex mutex;
    static std::map<std::pair<int, size_t>, int> known;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lock(mutex);
    const auto key = std::make_pair(dev, smem);
    const auto it = known.find(key);
    if (it != known.end()) return it->second;
    const Fp64ClusterKernel k = dr_fp64_cluster_kernel<true, 1>;
    prepare_fp64_cluster(k, smem);
    return known[key] = largest_cluster(k, smem);
}

// Dynamic shared memory of the allocation-free call's kernel: enough for every table
// of n nodes in `parts` pieces with n_elems elements, at most kSingleBytes.
constexpr size_t kSingleBytes = 200 * 1024;
static size_t single_bytes(int n, int n_elems, int parts) {
    const int m = (n + parts - 1) / parts;
    const Fp64Shape most = {parts, m, m, n_elems, 2 * n_elems, true, 1, false};
    return std::min(kSingleBytes, cluster_bytes(most));
}

cudaError_t prepare_dr_fp64_single(int *max_cluster) {
    cudaError_t e = cudaFuncSetAttribute(dr_fp64_single_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kSingleBytes);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(dr_fp64_single_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    *max_cluster = largest_cluster(dr_fp64_single_kernel, kSingleBytes);
    return *max_cluster > 0 ? cudaSuccess : cudaErrorLaunchOutOfResources;
}

int launch_dr_fp64_single(const DevMesh &m, const DevState &s, const DevResults &r, const SolveParams &p, int n,
                          int n_elems, int parts, const int *skip, const int32_t *perm, double *u, void *stream) {
    cudaLaunchAttribute attr[1];
    Fp64Shape sp = {};
    sp.parts = parts;
    cudaLaunchConfig_t cfg = fp64_cluster_config(1, sp, kMaxThreads, attr, static_cast<cudaStream_t>(stream));
    cfg.dynamicSmemBytes = single_bytes(n, n_elems, parts);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, dr_fp64_single_kernel, m, s, r, p, cfg.dynamicSmemBytes, skip, perm, u);
    if (e != cudaSuccess) return (int)e;
    return (int)cudaGetLastError();
}

}  // namespace fe2
