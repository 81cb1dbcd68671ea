// Internal device/host data layout of a batch (not part of the C ABI).
//
// Packed, CRS-like storage of many RVEs (the paper's PackedView: a row-offset
// vector plus value vectors holding every sub-problem of a rank contiguously,
// Section III), re-laid out for the GPU:
//   * nodes of RVE p occupy [node0, node0 + n_nodes) of every node array, free
//     nodes first (the paper's free/fixed reordering, Section III);
//   * an RVE is split spatially (recursive coordinate bisection) into
//     n_parts parts, one per CTA of the thread-block cluster that solves it in
//     mixed precision. Free nodes are ordered part by part (by degree within a
//     part), then fixed nodes part by part, so part r owns the free range
//     [part_f[r], part_f[r+1]) and the fixed range n_free + [part_g[r], part_g[r+1]);
//   * each node has a CSR row of its incident elements (node-centric, so the
//     force gather needs no atomics), ordered by the neighbour's ORIGINAL id:
//     the order in which a serial element scatter over lexicographic (a < b)
//     elements touches the node, which keeps FP64 sums bit-identical. `col`
//     holds the neighbour's RVE-local index, `col_part` the same neighbour as
//     (owning part << 16 | index inside that part's shared-memory arrays);
//   * structure-of-arrays per component for coalesced access.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace fe2 {

constexpr int kMaxParts = 16;  // largest (non-portable) thread-block cluster

struct RveDesc {
    int64_t node0;    // first node (permuted, global index)
    int64_t rp0;      // first row pointer: rowptr[rp0 .. rp0 + n_nodes]
    int64_t csr0;     // rowptr values are relative to this CSR entry
    int64_t elem0;    // first element of the stress list
    int32_t n_nodes;
    int32_t n_free;
    int32_t n_elems;
    int32_t n_parts;  // cluster size of the mixed solver for this RVE
    double dtc;       // critical time step (safety factor not applied)
    double c;         // damping coefficient
    double V0;        // reference volume
    int32_t part_max;       // largest part (nodes), sizes the shared memory
    int32_t part_free_max;  // most free nodes in one part
    int32_t part_elem_max;  // footprint rules: most elements with an end in one part
    int32_t part_slot_max;  // FP32 kernel: most row slots (ELL, 32-node slabs) of one part
    int64_t slot0;          // FP64 cluster kernel: first element slot of this RVE
    // FP64 cluster kernel: its parts (a multiple of n_parts), the largest of
    // them, and their most free nodes, element slots and row entries
    int32_t fp_parts;
    int32_t fp_part_max;
    int32_t fp_free_max;
    int32_t fp_slot_max;
    int32_t fp_row_max;
    int32_t fp_leaves;  // sets of nodes whose sums are formed first (a multiple of fp_parts)
    int32_t fp_groups;  // and the groups of each that are summed apart
    // FP32 phase of the mixed solver (dr_mixed_node.cu): most entries of a part's
    // increment array (free nodes, the zero entry, copies of other parts' nodes)
    // and most copies of its own nodes elsewhere; first copy; first global slot
    // of the rows that do not fit in shared memory
    int32_t part_q_max;
    int32_t part_push_max;
    int32_t part_u_max;   // lead: most entries of a part's displacement array
    int32_t ls_slot_max;  // lead: most element slots of a part
    int32_t flush_ok;  // lengths and rigidities far from FP32's limits (node_range_ok)
    int64_t ls_slot0;     // lead: first element slot
    int64_t push0;
    int64_t fix0;         // lead: first entry of lead_fix
    int64_t ell0;
};

// Launch shape of the FP64 cluster kernel: CTAs per cluster, capacities of one
// CTA, and what it keeps in shared memory beside the positions (tsm: element
// table and rows, ssm: the own free nodes' state, 1 with and 2 without their
// displacements, terms: the energy terms).
struct Fp64Shape {
    int parts, part_max, free_max, slot_max, row_max;
    bool tsm;
    int ssm;
    bool terms;
};
// CTAs per cluster of the FP32-phase kernel (dr_mixed_node.cu) and capacities of
// one CTA: increment entries, free nodes, row slots, copies of own nodes, and the row slots held in
// shared memory (the others are streamed from global memory).
struct NodeShape {
    int parts, q_cap, free_cap, slot_cap, push_cap, smem_slots;
    int alt;    // order of the fused operations in an element's force (entry_forces)
    int flush;  // RveDesc::flush_ok
};
// CTAs per cluster of the lead kernel (dr_mixed_lead.cu) and capacities of one
// CTA: displacement entries, free nodes, element slots, row entries (ELL), copies
// of own nodes; whether the part meets the footprint rule (staged) and whether
// the element constants are in shared memory.
struct LeadShape {
    int parts, u_cap, free_cap, elem_cap, slot_cap, push_cap;
    bool staged, ksm;
};

// Read-only, create-time arrays.
struct DevMesh {
    const RveDesc *rve;
    const double *X0, *X1, *X2;   // reference coordinates (permuted)
    const float *Xh, *Xl;         // reference coordinates as double-float, [3][N]
    const double *mass;           // lumped nodal mass
    const float *imh, *iml;       // 1/m as double-float
    const int32_t *rowptr;        // per RVE n_nodes + 1 entries
    const int32_t *col;           // neighbour (RVE-local permuted id)
    const int32_t *col_part;      // neighbour as (part << 16 | index in part)
    const int32_t *part_off;      // per RVE 2*(kMaxParts+1): part_f[], part_g[]
    const double *EA;             // per CSR entry
    const double *L;              // per CSR entry
    const float2 *eaf;            // per CSR entry: (EA, 1/L) double-float high parts
    const float2 *eaf_lo;         // per CSR entry: low parts
    const float4 *dh, *dl;        // per CSR entry: (X_j - X_i, L) as double-float hi / lo
    const int32_t *el_a, *el_b;   // stress elements (RVE-local permuted ids)
    const double *el_EA, *el_L;
    const int32_t *csr_el;        // per CSR entry: RVE-local element << 1, | 1 when
                                  // the row's node is the element's second node
                                  // (caller orientation)
    const int4 *fp_slot;          // FP64 cluster kernel and lead, per element slot: (element,
                                  // first end, second end, CSR entry << 1 | 1 when its row
                                  // is the second end's), ends as (part << 16 | index)
    const int32_t *fp_csr_slot;   // per row entry of a free node, in FP64 order from csr0:
                                  // part-relative slot << 1 | 1 when the node is the
                                  // element's second end
    const int32_t *fp_part_slot;  // per RVE kMaxParts+1 part slot offsets (from slot0)
    const int32_t *fp_node;       // FP64 order: RVE-local ids part by part, a part's free
                                  // nodes first, then its fixed ones
    const int32_t *fp_part_off;   // per RVE 2*(kMaxParts+1): the parts' first entries of
                                  // fp_node, and of the free nodes counted alone
    const int32_t *fp_row;        // per RVE n_free + 1 (from rp0): row offsets into
                                  // fp_csr_slot, free nodes in FP64 order
    const uint16_t *fp_leaf;      // the nodes again leaf by leaf, ascending RVE-local ids in a
                                  // leaf: index inside the part (null: a part is a leaf)
    const int32_t *fp_leaf_off;   // per RVE 2*(kMaxParts+1): the leaves' first entries of
                                  // fp_leaf (from node0), and each leaf's free nodes
    const int4 *ls_slot;          // lead: fp_slot, fp_csr_slot, fp_part_slot and fp_row by the
    const int32_t *ls_csr_slot;   // mixed solver's parts (the FP64 kernel's may divide them)
    const int32_t *ls_part_slot;
    const int32_t *ls_row;
    const uint16_t *qidx;         // FP32 phase, per CSR entry of a free node: the neighbour's
                                  // place in the part's increment array
    const int32_t *push_off;      // per RVE n_free + 1 (from rp0): copies of a free node in
                                  // other parts, offsets from push0
    const uint32_t *lead_ends;    // lead, per element slot (ls_slot): places of its ends in the
                                  // part's displacement array, first | second << 16
    const int32_t *lead_fix;      // lead: per part the fixed neighbours of its free nodes
                                  // (RVE-local ids, from fix0)
    const int32_t *lead_fix_off;  // per RVE 2*(kMaxParts+1): the parts' offsets into them, and
                                  // the place of each part's first in its displacement array
    const uint32_t *push;         // per copy: (part << 16 | place in its increment array)
};

// Mutable solver state (device). Its size places the kernel arguments behind it: one
// pointer more cost the FP32 phase of 5000-node RVEs 1.7 % (38.4 -> 39.1 ms for
// 20,000 iterations), two more saved it 0.9 % and cost 20,000-node RVEs 0.8 %.
struct DevState {
    double *u0, *u1, *u2;         // displacement (output of every mode)
    double *v0, *v1, *v2;         // FP64 velocity
    double *a0, *a1, *a2;         // FP64 acceleration; FP64 cluster kernel: kinetic
                                  // energies, and behind the three arrays those of two
                                  // more evaluations or the work terms, per RVE
                                  // [2][3][n] at 6 node0
    float *uh, *ul;               // MIXED: displacement, double-float [3][N]
    float *vh, *vl;               // MIXED: velocity (lead: double-float; FP32 phase: vh)
    float *ah, *al;               // MIXED: acceleration (same convention)
    float *fg;                    // MIXED: reference force g_ref, FP32 [3][N]
    double *xg;                   // [3][N] FP64 positions scratch
    double *tf;                   // FP64: per element, its force on the first node (3)
    float4 *sv;                   // MIXED FP32 kernel without tables: per node
    float2 *sa;                   //   (v, a.x) and (a.y, a.z)
    double *gp, *fdp;             // FP64 energy check: previous internal and damping
                                  // force per free DOF [3][N]
    double *ualt;                 // FP64 cluster kernel: displacements of the last three
                                  // evaluations, per RVE [3][3][n] at 9 node0, FP64 order;
                                  // FP32 phase: increments of the last four, float4 [4][n]
    float4 *ek0;                  // FP32 phase, row slots beyond shared memory: (r, EA)
    float *ek1;                   //   and q_ref
    double *fpt;                  // FP64 cluster kernel: element forces [3][part slots]
                                  // when the table does not fit in shared memory
};

struct DevResults {
    double *sigma;    // 9 per RVE
    int64_t *iters;
    double *rel_res;
    int32_t *status;
    double *f_ref;
    double *ke;
    int64_t *lead;    // MIXED: iterations run in the double-float lead
    double *wint;     // FP64 energy check: stored internal work since the start
    double *wext;     //   and work of the damping forces
};

struct SolveParams {
    const double *F;      // 9 per RVE (device)
    double tol;
    int64_t max_iter;
    double alpha;
    int init;
    int want_ke;          // 1: kinetic energy; 2 (FP64): also the work terms of the
                          // energy balance
    int64_t lead_iters;   // < 0: lead until the relative residual <= lead_tol
    double lead_tol;
    int rebase_every;
    const int32_t *queue; // RVE ids in scheduling order
    int32_t queue_len;
    int32_t *counter;     // work-queue heads (zeroed before the launch; mixed uses three)
    int smem_positions;   // FP64 kernel: 1 = positions staged in shared memory
    int64_t stall_window; // MIXED: FP32 evaluations without the squared residual
                          // falling to a quarter before the RVE is handed back
                          // to double-float; 0 = never
    int resume;           // MIXED lead kernel: 1 = resume launch (stalled RVEs only)
};

// RVE_STALLED (internal): the FP32 phase stopped making progress and the RVE
// waits for the double-float resume launch, which replaces the status.
enum { RVE_OK = 0, RVE_MAXITER = 1, RVE_NAN = 2, RVE_PENDING = 3, RVE_STALLED = 5 };
// Work-queue heads per launch class: lead, FP32 phase, double-float resume.
constexpr int kCountersPerClass = 3;

// Kernel launchers (defined in the .cu files).
int launch_setup(int32_t n_rve, int64_t n_el, int64_t n_csr, RveDesc *rve,
                 const int64_t *ga, const int64_t *gb, const double *X0, const double *X1,
                 const double *X2, const int64_t *elem_of, const double *EA_csr,
                 const double *el_EA, const int32_t *rowptr, double *el_L, double *L_csr,
                 float2 *eaf, float2 *eaf_lo, double *mass, float *imh, float *iml,
                 float *Xh, float *Xl, const int32_t *col, float4 *dh, float4 *dl,
                 void *stream);
int launch_dr_fp64(const DevMesh &m, const DevState &s, const DevResults &r,
                   const SolveParams &p, int grid, int block, size_t smem, void *stream);
// Mixed solver without tables (dr_mixed.cu): one thread-block cluster of `parts`
// CTAs per RVE; lead = 1 the double-float lead, 0 the FP32 phase.
int launch_dr_mixed(const DevMesh &m, const DevState &s, const DevResults &r,
                    const SolveParams &p, int lead, int clusters, int parts, int block,
                    size_t smem, int part_cap, void *stream);
// Footprint rules of the mixed solver (dr_mixed.cu): the bytes of a part with tables
// where they are within `limit`, else of its plain node state. The first sets the
// number of parts and the FP32 phase's order of operations, the second the lead's form.
size_t mixed_fp32_smem(int part_cap, int free_cap, int elem_cap, int slot_cap, size_t limit);
size_t mixed_lead_smem(int part_cap, int free_cap, int elem_cap, int slot_cap, size_t limit);
// Lead kernel (dr_mixed_lead.cu): dynamic shared memory, launch, co-resident
// clusters.
size_t lead_smem(const LeadShape &sp);
int launch_dr_mixed_lead(const DevMesh &m, const DevState &s, const DevResults &r, const SolveParams &p,
                         int clusters, int block, const LeadShape &sp, void *stream);
int occupancy_dr_mixed_lead(int block, const LeadShape &sp);
// FP32 phase with row tables (dr_mixed_node.cu): dynamic shared memory, launch,
// co-resident clusters.
size_t mixed_node_smem(const NodeShape &sp);
int launch_dr_mixed_node(const DevMesh &m, const DevState &s, const DevResults &r, const SolveParams &p,
                         int clusters, int block, size_t smem, const NodeShape &sp, bool pair, void *stream);
int occupancy_dr_mixed_node(int block, size_t smem, const NodeShape &sp, bool pair);
// Whether a footprint of `smem` bytes (by the rules above) is one with tables.
bool mixed_staged(int lead, size_t smem, int part_cap);
// FP64 cluster kernel (dr_fp64_cluster.cu): dynamic shared memory, launch,
// co-resident clusters. `block`: threads per CTA, the last warp of which tests
// the residual.
size_t fp64_cluster_smem(const Fp64Shape &sp);
int launch_dr_fp64_cluster(const DevMesh &m, const DevState &s, const DevResults &r, const SolveParams &p,
                           int clusters, int block, const Fp64Shape &sp, void *stream);
int occupancy_dr_fp64_cluster(int block, const Fp64Shape &sp);
// CTAs of the largest cluster of that kernel, each with smem bytes, that the device
// can hold.
int fp64_max_cluster(size_t smem);
// The same solver for the allocation-free call: one cluster of `parts` CTAs for
// RVE 0 of m (n nodes), tables in the caller's arrays; nothing to do when *skip.
cudaError_t prepare_dr_fp64_single(int *max_cluster);
int launch_dr_fp64_single(const DevMesh &m, const DevState &s, const DevResults &r, const SolveParams &p, int n,
                          int n_elems, int parts, const int *skip, const int32_t *perm, double *u, void *stream);
// Shared memory per node of a kernel without tables (dr_mixed.cu).
size_t mixed_plain_node_bytes(int lead);
// Resident CTAs per SM (FP64) / co-resident clusters (mixed) for a launch shape.
int occupancy_dr_fp64(int smem_positions, int block, size_t smem);
int occupancy_dr_mixed(int lead, int parts, int block, size_t smem);

// Naive comparator: scratch sized for the largest RVE, and one RVE's solve.
struct NaiveScratch {
    double *x, *g, *acc;  // 3*n_max, 3*n_max, 16
};
int naive_solve_rve(const RveDesc &R, const DevMesh &M, const DevState &S, const DevResults &O,
                    const double *F_dev, const NaiveScratch &W, double tol, int64_t max_iter,
                    double alpha, int init, int p, cudaStream_t st, int64_t *iters_out,
                    double *rel_out, int *status_out);

}  // namespace fe2
