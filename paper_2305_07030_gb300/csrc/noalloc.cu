// Allocation-free single-RVE solve: the FP64 oracle-order solver with all of
// its working memory in one file-scope device array.
//
// Some callers cannot call cudaMalloc: code that runs while a CUDA graph is
// being captured, real-time loops that must not allocate, or host frameworks
// that own every device allocation through their own pools. They hold their
// inputs and outputs in device memory they already have and need the library
// to allocate nothing. fe2_rve_solve_noalloc serves them with two launches: a
// packing kernel (one CTA) puts the RVE into the static scratch array below (node
// permutation, node-centric CSR, lumped masses, critical time step, a split of the
// nodes into spatially compact parts and each part's element slots), and the
// batched FP64 path's cluster kernel solves it, one part per CTA.
//
// The split follows the nodes' Morton order, cut into equal pieces: about the
// bisection's octants for evenly spread nodes, from one sort. The FP64 pipe of one
// SM (2 operations per clock) is what a one-CTA solve waits for: 700 nodes x 500
// iterations on one CTA 14.3 ms, on 16 CTAs 1.95; 4000 nodes on 8 CTAs 18.4 us per
// iteration, on 16 13.2.
//
// The scratch array is shared by every call on a device and keeps the last
// call's contents; everything a solve reads is rewritten or cleared by that
// solve. Calls whose work overlaps on the GPU race on it. The array occupies
// kNoallocScratchBytes of device memory on every GPU that loads the library,
// until the process exits.
#include <cuda_runtime.h>

#include <mutex>
#include <string>

#include "../../include/fe2.h"
#include "dr_device.cuh"
#include "fp64_parts.h"

namespace fe2 {
namespace {

constexpr int kNaMaxNodes = 4096;
constexpr int kNaMaxElems = 16384;
constexpr int kNaThreads = 512;

// Byte layout of the scratch array (every block 256-byte aligned).
constexpr size_t align256(size_t x) { return (x + 255) & ~size_t(255); }
constexpr size_t kOffRve = 0;
constexpr size_t kOffX = align256(kOffRve + sizeof(RveDesc));
constexpr size_t kOffMass = align256(kOffX + sizeof(double) * 3 * kNaMaxNodes);
constexpr size_t kOffU = align256(kOffMass + sizeof(double) * kNaMaxNodes);
constexpr size_t kOffV = align256(kOffU + sizeof(double) * 3 * kNaMaxNodes);
constexpr size_t kOffA = align256(kOffV + sizeof(double) * 3 * kNaMaxNodes);
constexpr size_t kOffRow = align256(kOffA + sizeof(double) * 3 * kNaMaxNodes);
constexpr size_t kOffCol = align256(kOffRow + sizeof(int32_t) * (kNaMaxNodes + 1));
constexpr size_t kOffElemOf = align256(kOffCol + sizeof(int32_t) * 2 * kNaMaxElems);
constexpr size_t kOffEAc = align256(kOffElemOf + sizeof(int32_t) * 2 * kNaMaxElems);
constexpr size_t kOffLc = align256(kOffEAc + sizeof(double) * 2 * kNaMaxElems);
constexpr size_t kOffElA = align256(kOffLc + sizeof(double) * 2 * kNaMaxElems);
constexpr size_t kOffElB = align256(kOffElA + sizeof(int32_t) * kNaMaxElems);
constexpr size_t kOffElEA = align256(kOffElB + sizeof(int32_t) * kNaMaxElems);
constexpr size_t kOffElL = align256(kOffElEA + sizeof(double) * kNaMaxElems);
constexpr size_t kOffPerm = align256(kOffElL + sizeof(double) * kNaMaxElems);  // permuted -> caller
constexpr size_t kOffInv = align256(kOffPerm + sizeof(int32_t) * kNaMaxNodes);  // caller -> permuted
constexpr size_t kOffDeg = align256(kOffInv + sizeof(int32_t) * kNaMaxNodes);
constexpr size_t kOffCur = align256(kOffDeg + sizeof(int32_t) * kNaMaxNodes);
constexpr size_t kOffMisc = align256(kOffCur + sizeof(int32_t) * kNaMaxNodes);  // f_ref, ke, skip flag
// FP64 cluster kernel: displacement ring, element forces, slots and rows by part
constexpr size_t kOffRing = align256(kOffMisc + 3 * sizeof(double));
constexpr size_t kOffForce = align256(kOffRing + sizeof(double) * 9 * kNaMaxNodes);
constexpr size_t kOffSlot = align256(kOffForce + sizeof(double) * 3 * 2 * kNaMaxElems);
constexpr size_t kOffCsrSlot = align256(kOffSlot + sizeof(int4) * 2 * kNaMaxElems);
constexpr size_t kOffSlotA = align256(kOffCsrSlot + sizeof(int32_t) * 2 * kNaMaxElems);  // per element: slot in its
constexpr size_t kOffSlotB = align256(kOffSlotA + sizeof(int32_t) * kNaMaxElems);        // first / second end's part
constexpr size_t kOffPartSlot = align256(kOffSlotB + sizeof(int32_t) * kNaMaxElems);
constexpr size_t kOffNode = align256(kOffPartSlot + sizeof(int32_t) * (kMaxParts + 1));
constexpr size_t kOffRef = align256(kOffNode + sizeof(int32_t) * kNaMaxNodes);   // (part << 16 | index in part)
constexpr size_t kOffPartOff = align256(kOffRef + sizeof(int32_t) * kNaMaxNodes);
constexpr size_t kOffFrow = align256(kOffPartOff + sizeof(int32_t) * 2 * (kMaxParts + 1));
constexpr size_t kOffKin = align256(kOffFrow + sizeof(int32_t) * (kNaMaxNodes + 1));  // kinetic energies
constexpr size_t kNoallocScratchBytes = align256(kOffKin + sizeof(double) * 9 * kNaMaxNodes);

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocScratchBytes];

// Per-RVE status written when the device-side input checks fail.
constexpr int kRveInvalid = 4;

struct NaArgs {
    int n, E;
    const double *X;       // caller, 3n xyz interleaved
    const int32_t *conn;   // caller, 2E local ids
    const double *EA;      // caller, E
    const uint8_t *fixed;  // caller, n
    const double *F;       // caller, 9
    double c, V0;
    double *u;             // caller, 3n (input for warm start, output)
    double *sigma;         // caller, 9
    int64_t *iters;        // caller, 1
    double *rel_res;       // caller, 1
    int32_t *status;       // caller, 1
};

__device__ __forceinline__ int block_excl_scan(int v, int *tmp) {
    // exclusive scan over the CTA (kNaThreads threads, 16 warps)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) tmp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int w = lane < (kNaThreads >> 5) ? tmp[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        if (lane < (kNaThreads >> 5)) tmp[lane] = w;
    }
    __syncthreads();
    const int before = warp > 0 ? tmp[warp - 1] : 0;
    __syncthreads();
    return before + x - v;
}

// 10 bits of x spread to every third bit.
__device__ __forceinline__ uint32_t spread3(uint32_t x) {
    x = (x | (x << 16)) & 0x030000ffu;
    x = (x | (x << 8)) & 0x0300f00fu;
    x = (x | (x << 4)) & 0x030c30c3u;
    return (x | (x << 2)) & 0x09249249u;
}

__global__ void __launch_bounds__(kNaThreads) k_noalloc_pack(NaArgs A, int warm, int C, int groups, unsigned char *scr) {
    extern __shared__ __align__(16) uint64_t keys[];  // the next power of two above n
    __shared__ double red[6 * (kNaThreads / 32)];
    __shared__ int tmp[32];
    __shared__ int err, nfree_s;
    RveDesc *rve = reinterpret_cast<RveDesc *>(scr + kOffRve);
    double *X = reinterpret_cast<double *>(scr + kOffX);
    double *mass = reinterpret_cast<double *>(scr + kOffMass);
    double *u = reinterpret_cast<double *>(scr + kOffU);
    int32_t *row = reinterpret_cast<int32_t *>(scr + kOffRow);
    int32_t *col = reinterpret_cast<int32_t *>(scr + kOffCol);
    int32_t *elem_of = reinterpret_cast<int32_t *>(scr + kOffElemOf);
    double *EAc = reinterpret_cast<double *>(scr + kOffEAc);
    double *Lc = reinterpret_cast<double *>(scr + kOffLc);
    int32_t *el_a = reinterpret_cast<int32_t *>(scr + kOffElA);
    int32_t *el_b = reinterpret_cast<int32_t *>(scr + kOffElB);
    double *el_EA = reinterpret_cast<double *>(scr + kOffElEA);
    double *el_L = reinterpret_cast<double *>(scr + kOffElL);
    int32_t *perm = reinterpret_cast<int32_t *>(scr + kOffPerm);
    int32_t *inv = reinterpret_cast<int32_t *>(scr + kOffInv);
    int32_t *deg = reinterpret_cast<int32_t *>(scr + kOffDeg);
    int32_t *cur = reinterpret_cast<int32_t *>(scr + kOffCur);
    int *skip = reinterpret_cast<int *>(scr + kOffMisc + 2 * sizeof(double));
    const int n = A.n, E = A.E;

    // ---- checks of the device-side inputs; degrees ----
    if (threadIdx.x == 0) {
        err = 0;
        *skip = 1;  // until the tables are complete
    }
    __syncthreads();  // the flag is clear before any thread may set it
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        deg[i] = 0;
        const double *x = A.X + 3 * i;
        if (!isfinite(x[0]) || !isfinite(x[1]) || !isfinite(x[2])) err = 1;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < E; e += blockDim.x) {
        const int p = A.conn[2 * e], q = A.conn[2 * e + 1];
        if (p < 0 || q < 0 || p >= n || q >= n || p == q || !(A.EA[e] > 0.0) || !isfinite(A.EA[e])) {
            err = 1;
            continue;
        }
        const double *xp = A.X + 3 * p, *xq = A.X + 3 * q;
        if (xp[0] == xq[0] && xp[1] == xq[1] && xp[2] == xq[2]) err = 1;
        atomicAdd(deg + p, 1);
        atomicAdd(deg + q, 1);
    }
    __syncthreads();
    if (err) {
        if (threadIdx.x == 0) {
            *A.status = kRveInvalid;
            *A.iters = 0;
            *A.rel_res = 0.0;
        }
        return;
    }

    // ---- permutation: free nodes first, then fixed, each in caller order ----
    // (a free node that no element touches is held fixed)
    constexpr int kPer = kNaMaxNodes / kNaThreads;
    int fl[kPer], cnt = 0;
    for (int k = 0; k < kPer; ++k) {
        const int i = threadIdx.x * kPer + k;
        fl[k] = (i < n && !A.fixed[i] && deg[i] > 0) ? 1 : 0;
        cnt += fl[k];
    }
    int off = block_excl_scan(cnt, tmp);
    if (threadIdx.x == blockDim.x - 1) nfree_s = off + cnt;
    __syncthreads();
    const int nf = nfree_s;
    int offx = block_excl_scan((threadIdx.x * kPer < n ? min(kPer, n - (int)threadIdx.x * kPer) : 0) - cnt, tmp);
    for (int k = 0; k < kPer; ++k) {
        const int i = threadIdx.x * kPer + k;
        if (i >= n) break;
        const int pi = fl[k] ? off++ : nf + offx++;
        perm[pi] = i;
        inv[i] = pi;
    }
    __syncthreads();

    // ---- node-centric CSR: row pointers, entries, rows sorted by caller id ----
    int dsum = 0;
    for (int k = 0; k < kPer; ++k) {
        const int pi = threadIdx.x * kPer + k;
        if (pi < n) dsum += deg[perm[pi]];
    }
    int roff = block_excl_scan(dsum, tmp);
    for (int k = 0; k < kPer; ++k) {
        const int pi = threadIdx.x * kPer + k;
        if (pi < n) {
            row[pi] = roff;
            cur[pi] = roff;
            roff += deg[perm[pi]];
        }
    }
    if (threadIdx.x == 0) row[n] = 2 * E;
    __syncthreads();
    for (int e = threadIdx.x; e < E; e += blockDim.x) {
        const int p = inv[A.conn[2 * e]], q = inv[A.conn[2 * e + 1]];
        const int sp = atomicAdd(cur + p, 1), sq = atomicAdd(cur + q, 1);
        col[sp] = q; elem_of[sp] = e;
        col[sq] = p; elem_of[sq] = e;
    }
    __syncthreads();
    for (int pi = threadIdx.x; pi < n; pi += blockDim.x) {
        const int b = row[pi], en = row[pi + 1];
        for (int s = b + 1; s < en; ++s) {  // insertion sort by caller id of the neighbour
            const int cj = col[s], ej = elem_of[s], key = perm[cj];
            int t = s - 1;
            while (t >= b && perm[col[t]] > key) {
                col[t + 1] = col[t];
                elem_of[t + 1] = elem_of[t];
                --t;
            }
            col[t + 1] = cj;
            elem_of[t + 1] = ej;
        }
        for (int s = b + 1; s < en; ++s)
            if (col[s] == col[s - 1]) err = 1;  // repeated element
    }
    __syncthreads();
    if (err) {
        if (threadIdx.x == 0) {
            *A.status = kRveInvalid;
            *A.iters = 0;
            *A.rel_res = 0.0;
        }
        return;
    }

    // ---- coordinates, lengths, masses, stress elements, time step ----
    for (int pi = threadIdx.x; pi < n; pi += blockDim.x) {
        const int i = perm[pi];
        for (int c = 0; c < 3; ++c) X[c * n + pi] = A.X[3 * i + c];
    }
    for (int e = threadIdx.x; e < E; e += blockDim.x) {
        const int p = A.conn[2 * e], q = A.conn[2 * e + 1];
        const double *xp = A.X + 3 * p, *xq = A.X + 3 * q;
        const double dx = dsub(xq[0], xp[0]), dy = dsub(xq[1], xp[1]), dz = dsub(xq[2], xp[2]);
        el_L[e] = dsqrt(dadd(dadd(dmul(dx, dx), dmul(dy, dy)), dmul(dz, dz)));
        el_a[e] = inv[p];
        el_b[e] = inv[q];
        el_EA[e] = A.EA[e];
    }
    __syncthreads();
    for (int s = threadIdx.x; s < 2 * E; s += blockDim.x) {
        EAc[s] = A.EA[elem_of[s]];
        Lc[s] = el_L[elem_of[s]];
    }
    __syncthreads();
    for (int pi = threadIdx.x; pi < n; pi += blockDim.x) {
        double m = 0.0;
        for (int s = row[pi]; s < row[pi + 1]; ++s) {
            const double L = Lc[s];
            const double rhoA = ddiv(EAc[s], dmul(L, L));
            m = dadd(m, dmul(0.5, dmul(rhoA, L)));
        }
        mass[pi] = m;
        // warm start reads the caller's displacement (caller order)
        for (int c = 0; c < 3; ++c) u[c * n + pi] = warm ? A.u[3 * perm[pi] + c] : 0.0;
    }
    double tmin = INFINITY;
    for (int e = threadIdx.x; e < E; e += blockDim.x) {
        const double L = el_L[e], EA = el_EA[e];
        const double rhoA = ddiv(EA, dmul(L, L));
        const double t = dmul(L, dsqrt(ddiv(rhoA, EA)));
        tmin = t < tmin ? t : tmin;
    }
    for (int o = 16; o > 0; o >>= 1) {
        const double other = __shfl_xor_sync(0xffffffffu, tmin, o);
        tmin = other < tmin ? other : tmin;
    }
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = tmin;
    __syncthreads();
    __shared__ double dtc;
    if (threadIdx.x == 0) {
        double t = INFINITY;
        for (int w = 0; w < (kNaThreads >> 5); ++w) t = red[w] < t ? red[w] : t;
        dtc = t;
    }
    __syncthreads();

    // ---- Morton order of the nodes ----
    double lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (int pi = threadIdx.x; pi < n; pi += blockDim.x)
        for (int c = 0; c < 3; ++c) {
            lo[c] = fmin(lo[c], X[c * n + pi]);
            hi[c] = fmax(hi[c], X[c * n + pi]);
        }
    for (int c = 0; c < 3; ++c) {
        for (int o = 16; o > 0; o >>= 1) {
            lo[c] = fmin(lo[c], __shfl_xor_sync(0xffffffffu, lo[c], o));
            hi[c] = fmax(hi[c], __shfl_xor_sync(0xffffffffu, hi[c], o));
        }
        if ((threadIdx.x & 31) == 0) {
            red[6 * (threadIdx.x >> 5) + c] = lo[c];
            red[6 * (threadIdx.x >> 5) + 3 + c] = hi[c];
        }
    }
    __syncthreads();
    for (int c = 0; c < 3; ++c)
        for (int w = 0; w < (kNaThreads >> 5); ++w) {
            lo[c] = fmin(lo[c], red[6 * w + c]);
            hi[c] = fmax(hi[c], red[6 * w + 3 + c]);
        }
    int np = 1;
    while (np < n) np *= 2;
    for (int i = threadIdx.x; i < np; i += blockDim.x) {
        uint32_t code = 0;
        if (i < n && C > 1)
            for (int c = 0; c < 3; ++c) {
                const double w = hi[c] - lo[c];
                const double f = w > 0.0 ? (X[c * n + i] - lo[c]) / w : 0.0;
                code |= spread3((uint32_t)min(1023, max(0, (int)(f * 1024.0)))) << c;
            }
        keys[i] = i < n ? ((uint64_t)code << 32) | (uint32_t)i : ~0ull;
    }
    __syncthreads();
    if (C > 1)  // bitonic sort
        for (int k = 2; k <= np; k *= 2)
            for (int j = k / 2; j > 0; j /= 2) {
                for (int i = threadIdx.x; i < np; i += blockDim.x) {
                    const int x = i ^ j;
                    if (x > i) {
                        const uint64_t ki = keys[i], kx = keys[x];
                        if ((ki > kx) == ((i & k) == 0)) {
                            keys[i] = kx;
                            keys[x] = ki;
                        }
                    }
                }
                __syncthreads();
            }

    // ---- parts: equal pieces of that order, a part's free nodes first ----
    int4 *slot = reinterpret_cast<int4 *>(scr + kOffSlot);
    int32_t *csr_slot = reinterpret_cast<int32_t *>(scr + kOffCsrSlot);
    int32_t *slot_a = reinterpret_cast<int32_t *>(scr + kOffSlotA), *slot_b = reinterpret_cast<int32_t *>(scr + kOffSlotB);
    int32_t *part_slot = reinterpret_cast<int32_t *>(scr + kOffPartSlot);
    int32_t *node = reinterpret_cast<int32_t *>(scr + kOffNode), *ref = reinterpret_cast<int32_t *>(scr + kOffRef);
    int32_t *part_off = reinterpret_cast<int32_t *>(scr + kOffPartOff), *part_free = part_off + kMaxParts + 1;
    int32_t *frow = reinterpret_cast<int32_t *>(scr + kOffFrow);
    auto first = [&](int r) { return (int)((int64_t)r * n / C); };  // a part's first place in the order
    // free nodes before each place (into cur; nf at the end is part_free[C])
    cnt = 0;
    for (int k = 0; k < kPer; ++k) {
        const int q = threadIdx.x * kPer + k;
        cnt += q < n && (int)(uint32_t)keys[q] < nf;
    }
    off = block_excl_scan(cnt, tmp);
    for (int k = 0; k < kPer; ++k) {
        const int q = threadIdx.x * kPer + k;
        if (q >= n) break;
        cur[q] = off;
        off += (int)(uint32_t)keys[q] < nf;
    }
    __syncthreads();
    for (int r = threadIdx.x; r <= kMaxParts; r += blockDim.x) {
        part_off[r] = r < C ? first(r) : n;
        part_free[r] = r < C && first(r) < n ? cur[first(r)] : nf;
    }
    __syncthreads();
    for (int q = threadIdx.x; q < n; q += blockDim.x) {
        const int pi = (int)(uint32_t)keys[q];
        int r = 0;
        while (r + 1 < C && q >= part_off[r + 1]) ++r;
        const int fi = cur[q] - part_free[r], nfr = part_free[r + 1] - part_free[r];
        const int idx = pi < nf ? fi : nfr + (q - part_off[r]) - fi;
        ref[pi] = (r << 16) | idx;
        node[part_off[r] + idx] = pi;
        if (pi < nf) deg[cur[q]] = row[pi + 1] - row[pi];  // row lengths in part order
    }
    __syncthreads();
    dsum = 0;
    for (int k = 0; k < kPer; ++k) {
        const int x = threadIdx.x * kPer + k;
        if (x < nf) dsum += deg[x];
    }
    roff = block_excl_scan(dsum, tmp);
    for (int k = 0; k < kPer; ++k) {
        const int x = threadIdx.x * kPer + k;
        if (x < nf) {
            frow[x] = roff;
            roff += deg[x];
            if (x == nf - 1) frow[nf] = roff;
        }
    }
    if (threadIdx.x == 0 && nf == 0) frow[0] = 0;

    // ---- element slots: per part, the elements with an end among its free nodes ----
    const int per = (E + kNaThreads - 1) / kNaThreads, eb = min(E, (int)threadIdx.x * per), ee = min(E, eb + per);
    int base = 0, slot_max = 0;
    __shared__ int total;
    for (int r = 0; r < C; ++r) {
        auto mine = [&](int p) { return p < nf && (ref[p] >> 16) == r; };
        int m = 0;
        for (int e = eb; e < ee; ++e) m += mine(el_a[e]) || mine(el_b[e]);
        int at = block_excl_scan(m, tmp);
        if (threadIdx.x == kNaThreads - 1) total = at + m;
        for (int e = eb; e < ee; ++e) {
            const int p = el_a[e], q = el_b[e];
            const bool ma = mine(p), mb = mine(q);
            if (!ma && !mb) continue;
            if (ma) slot_a[e] = at;
            if (mb) slot_b[e] = at;
            slot[base + at++] = make_int4(e, ref[p], ref[q], 0);
        }
        __syncthreads();
        if (threadIdx.x == 0) part_slot[r] = base;
        base += total;
        slot_max = max(slot_max, total);
        __syncthreads();
    }
    if (threadIdx.x == 0)
        for (int r = C; r <= kMaxParts; ++r) part_slot[r] = base;
    __syncthreads();
    for (int pi = threadIdx.x; pi < nf; pi += blockDim.x) {
        const int w = ref[pi], x = part_free[w >> 16] + (w & 0xffff);
        for (int q = row[pi], o = frow[x]; q < row[pi + 1]; ++q, ++o) {
            const int e = elem_of[q], second = el_b[e] == pi;
            csr_slot[o] = ((second ? slot_b[e] : slot_a[e]) << 1) | second;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        RveDesc R = {};
        R.n_nodes = n; R.n_free = nf; R.n_elems = E; R.n_parts = C;
        R.dtc = dtc; R.c = A.c; R.V0 = A.V0;
        R.fp_parts = R.fp_leaves = C;
        R.fp_groups = groups;
        R.fp_slot_max = slot_max;
        for (int r = 0; r < C; ++r) {
            R.fp_part_max = max(R.fp_part_max, part_off[r + 1] - part_off[r]);
            R.fp_free_max = max(R.fp_free_max, part_free[r + 1] - part_free[r]);
            R.fp_row_max = max(R.fp_row_max, frow[part_free[r + 1]] - frow[part_free[r]]);
        }
        *rve = R;
        *skip = 0;
    }
}

std::mutex g_na_mutex;
void *g_na_ptr[64] = {};
int g_na_cluster[64] = {};  // largest cluster of the solver's kernel; 0: not yet known
thread_local std::string g_na_err;

}  // namespace
}  // namespace fe2

using namespace fe2;

extern "C" const char *fe2_noalloc_last_error(void) { return g_na_err.c_str(); }

extern "C" size_t fe2_noalloc_scratch_bytes(void) { return kNoallocScratchBytes; }

extern "C" fe2_status fe2_rve_solve_noalloc(int32_t n_nodes, int32_t n_elems, const double *X_dev,
                                            const int32_t *conn_dev, const double *EA_dev,
                                            const uint8_t *fixed_dev, const double *F_dev,
                                            double damping, double V0, const fe2_opts *opts,
                                            double *u_dev, double *sigma_dev, int64_t *iters_dev,
                                            double *rel_res_dev, int32_t *status_dev,
                                            void *stream) {
    if (n_nodes < 1 || n_nodes > kNaMaxNodes) {
        g_na_err = "n_nodes must be in [1, " + std::to_string(kNaMaxNodes) + "]";
        return FE2_EINVAL;
    }
    if (n_elems < 0 || n_elems > kNaMaxElems) {
        g_na_err = "n_elems must be in [0, " + std::to_string(kNaMaxElems) + "]";
        return FE2_EINVAL;
    }
    if (!X_dev || !fixed_dev || !F_dev || !u_dev || !sigma_dev || !iters_dev || !rel_res_dev ||
        !status_dev || (n_elems > 0 && (!conn_dev || !EA_dev))) {
        g_na_err = "NULL device pointer";
        return FE2_EINVAL;
    }
    fe2_opts o;
    if (opts) o = *opts; else fe2_opts_default(&o);
    if (o.precision != FE2_PREC_FP64) {
        g_na_err = "the allocation-free entry point runs the FP64 solver only";
        return FE2_EINVAL;
    }
    if (!(o.tol >= 0.0) || o.max_iter < 1 || !(o.dt_safety > 0.0 && o.dt_safety <= 1.0) ||
        o.init < 0 || o.init > 2) {
        g_na_err = "invalid options";
        return FE2_EINVAL;
    }
    if (!(V0 > 0.0)) {
        g_na_err = "V0 must be > 0";
        return FE2_EINVAL;
    }
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= 64) {
        g_na_err = std::string("cudaGetDevice: ") + cudaGetErrorString(e);
        return FE2_ECUDA;
    }
    void *scratch = nullptr;
    int max_cluster = 0;
    {
        // once per device, with that device current: the device address of the
        // scratch array (its name in host code is not a device address)
        std::lock_guard<std::mutex> lock(g_na_mutex);
        if (!g_na_ptr[dev]) {
            e = cudaGetSymbolAddress(&g_na_ptr[dev], g_noalloc_scratch);
            if (e != cudaSuccess) {
                g_na_ptr[dev] = nullptr;
                g_na_err = std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e);
                return FE2_ECUDA;
            }
        }
        if (!g_na_cluster[dev]) {
            e = prepare_dr_fp64_single(&g_na_cluster[dev]);
            if (e != cudaSuccess) {
                g_na_cluster[dev] = 0;
                g_na_err = std::string("solver kernel: ") + cudaGetErrorString(e);
                return FE2_ECUDA;
            }
        }
        max_cluster = g_na_cluster[dev];
        scratch = g_na_ptr[dev];
    }
    NaArgs A;
    A.n = n_nodes;
    A.E = n_elems;
    A.X = X_dev;
    A.conn = conn_dev;
    A.EA = EA_dev;
    A.fixed = fixed_dev;
    A.F = F_dev;
    A.c = damping >= 0.0 ? damping : 0.002 * cbrt(512.0 / (double)n_nodes);
    A.V0 = V0;
    A.u = u_dev;
    A.sigma = sigma_dev;
    A.iters = iters_dev;
    A.rel_res = rel_res_dev;
    A.status = status_dev;
    SolveParams P = {};
    P.F = F_dev;
    P.tol = o.tol;
    P.max_iter = o.max_iter;
    P.alpha = o.dt_safety;
    P.init = o.init;
    P.want_ke = o.kinetic_energy != 0 ? 1 : 0;  // kinetic energy only: no work-sum scratch here
    unsigned char *scr = static_cast<unsigned char *>(scratch);
    const int n = n_nodes, C = fp64_single_parts(n, max_cluster);
    int np = 1;
    while (np < n) np *= 2;
    k_noalloc_pack<<<1, kNaThreads, sizeof(uint64_t) * np, static_cast<cudaStream_t>(stream)>>>(A, o.init == 2, C, fp64_groups(n, C, C),
                                                                                               scr);
    e = cudaGetLastError();
    if (e != cudaSuccess) {
        g_na_err = std::string("launch: ") + cudaGetErrorString(e);
        return FE2_ECUDA;
    }
    auto D = [&](size_t at) { return reinterpret_cast<double *>(scr + at); };
    auto I = [&](size_t at) { return reinterpret_cast<int32_t *>(scr + at); };
    DevMesh M = {};
    M.rve = reinterpret_cast<RveDesc *>(scr + kOffRve);
    M.X0 = D(kOffX); M.X1 = M.X0 + n; M.X2 = M.X0 + 2 * n;
    M.mass = D(kOffMass);
    M.rowptr = I(kOffRow);
    M.col = I(kOffCol);
    M.EA = D(kOffEAc);
    M.L = D(kOffLc);
    M.el_a = I(kOffElA); M.el_b = I(kOffElB); M.el_EA = D(kOffElEA); M.el_L = D(kOffElL);
    M.fp_slot = reinterpret_cast<int4 *>(scr + kOffSlot);
    M.fp_csr_slot = I(kOffCsrSlot);
    M.fp_part_slot = I(kOffPartSlot);
    M.fp_node = I(kOffNode);
    M.fp_part_off = I(kOffPartOff);
    M.fp_row = I(kOffFrow);
    DevState S = {};
    S.u0 = D(kOffU); S.u1 = S.u0 + n; S.u2 = S.u0 + 2 * n;
    S.v0 = D(kOffV); S.v1 = S.v0 + n; S.v2 = S.v0 + 2 * n;
    S.xg = D(kOffA);
    S.a0 = D(kOffKin); S.a1 = S.a0 + n; S.a2 = S.a0 + 2 * n;
    S.ualt = D(kOffRing);
    S.fpt = D(kOffForce);
    DevResults O = {};
    O.sigma = A.sigma; O.iters = A.iters; O.rel_res = A.rel_res; O.status = A.status;
    O.f_ref = D(kOffMisc); O.ke = D(kOffMisc) + 1;
    e = (cudaError_t)launch_dr_fp64_single(M, S, O, P, n, n_elems, C, reinterpret_cast<int *>(scr + kOffMisc + 2 * sizeof(double)),
                                           I(kOffPerm), A.u, stream);
    if (e != cudaSuccess) {
        g_na_err = std::string("launch: ") + cudaGetErrorString(e);
        return FE2_ECUDA;
    }
    return FE2_OK;
}
