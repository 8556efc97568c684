// Internal declarations of libsta: context layout, device helpers shared by the fold
// kernels, launch helpers.  Not part of the public ABI (see include/sta.h).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "sta.h"

namespace sta {

// ------------------------------------------------------------------------------------
// Error plumbing
// ------------------------------------------------------------------------------------
void set_error(const std::string &msg);
int fail(int code, const std::string &msg);

#define STA_CUDA_TRY(expr)                                                                   \
    do {                                                                                     \
        cudaError_t _e = (expr);                                                             \
        if (_e != cudaSuccess)                                                               \
            return ::sta::fail(_e == cudaErrorMemoryAllocation ? STA_ENOMEM : STA_ECUDA,     \
                               std::string(#expr) + ": " + cudaGetErrorString(_e));         \
    } while (0)

#define STA_TRY(expr)                                                                        \
    do {                                                                                     \
        int _s = (expr);                                                                     \
        if (_s != STA_OK) return _s;                                                         \
    } while (0)

// ------------------------------------------------------------------------------------
// Element cache: the 78 unique entries of each symmetric 12x12 element matrix, grouped by 3x3
// node-pair block into runs
//   diagonal block (a, a): 6 doubles, entries i <= j row-major (0,0) (0,1) (0,2) (1,1) (1,2) (2,2)
//   pair block (a, b), a < b local indices: 9 doubles, the block row-major over the node with the
//                          LOWER global id, i.e. K[3a+i][3b+j] at 3i+j if id(a) < id(b), else at 3j+i
// and stored by fold unit (node pair), not by tetrahedron: unit u's runs follow one another from
// Ke[bmeta[u].z] in ascending tetrahedron id, the order in which a fold adds them, every unit from
// an even offset (16 bytes).  So a fold needs no list of addresses -- its j-th contributor's run
// is at a fixed stride -- and reads its operands as one contiguous piece; which contributors are
// active is a bit each (UnitState).  Oriented by node id, a run is read as is (the folds never
// transpose).  krun[10 t + s] is the offset of tet t's run of unit slot s.
// ------------------------------------------------------------------------------------
constexpr int KE_STRIDE = 84;  // doubles of the cache per tetrahedron at most (4 x 6 + 6 x (9 + pad))
constexpr int RUN_DIAG = 6, RUN_PAIR = 9;

// index of (i, j), i <= j, inside a diagonal 6-run
__host__ __device__ inline int ke_tri(int i, int j) {
    return i == 0 ? j : (i == 1 ? 2 + j : 5);
}

// Contributor code of a fold unit (node pair a <= b) while the lists are built: tetrahedron id and
// the local indices of the unit's nodes a (la) and b (lb) inside that tetrahedron.
__host__ __device__ inline int32_t contrib_code(int32_t t, int la, int lb) {
    return (t << 4) | (la << 2) | lb;
}
__host__ __device__ inline int32_t code_tet(int32_t code) { return (code >> 4) & 0x07ffffff; }

// Activity of a unit's contributors, kept equal to the mask by every call that changes it, and the
// claims of the streaming frame in progress.  Contributor j's bit: w0 bit j (j < 32), w1 bit j - 32
// (j < 64), else bit j % 32 of uext[xoff + j / 32 - 2].  w0 and claims are one 64-bit word to the
// claim kernels (claim_unit); the thread that finds no claim yet has won the unit.  claims is 0 between
// frames.
struct __align__(16) UnitState {
    uint32_t w0, claims, w1, xoff;  // xoff: UNIT_NARROW for at most 64 contributors
};
constexpr uint32_t UNIT_NARROW = 0xffffffffu;

// The 10 unit slots of a tetrahedron: 0..3 diagonal (la, la), 4..9 the pairs (0,1) (0,2) (0,3)
// (1,2) (1,3) (2,3).
__host__ __device__ inline int slot_la(int s) { return s < 4 ? s : (s < 7 ? 0 : (s < 9 ? 1 : 2)); }
__host__ __device__ inline int slot_lb(int s) {
    return s < 4 ? s : (s == 4 ? 1 : (s == 5 ? 2 : (s == 6 ? 3 : (s == 7 ? 2 : 3))));
}
__host__ __device__ inline int slot_of(int la, int lb) {  // unordered local pair -> slot
    if (la == lb) return la;
    const int lo = la < lb ? la : lb, hi = la < lb ? lb : la;
    return 4 + (lo == 0 ? hi - 1 : (lo == 1 ? hi + 1 : 5));
}

// Units of one chunk of the rebuild fold -- their entries (9 per pair unit, 6 per diagonal unit) are
// whole rounds of 32 lanes, the last one nearly -- and the bytes of their runs.
constexpr int CHUNK_PAIR = 28, CHUNK_DIAG = 16, CHUNK_BYTES = 12 * 1024;

// Frame block: what one streaming frame brings -- the edited count and, right after the header, the
// edited list (tet id | new state << 31).  A frame's counters: [1] touched units (the FP64 re-fold
// counts them as diagonal | pair << 32), [3] touched CSR entries.
struct FrameHeader {
    int64_t m;                     // edited tetrahedra
    int64_t pad[3];
};
static_assert(sizeof(FrameHeader) == 32, "frame header layout");
inline int32_t *frame_edited(FrameHeader *f) { return reinterpret_cast<int32_t *>(f + 1); }
inline size_t frame_bytes(int64_t m) { return sizeof(FrameHeader) + sizeof(int32_t) * (size_t)m; }

// ------------------------------------------------------------------------------------
// Context
// ------------------------------------------------------------------------------------
// Operator of a context: the elasticity operator (sta_create, sta_batch_create) or the
// graph-Laplacian proxy (sta_proxy_create).
constexpr int STA_OP_ELASTICITY = 0;
constexpr int STA_OP_PROXY = 1;

// What a solve leaves for the host.
struct CgResult {
    double rr, bb;       // ||r||^2 at exit, ||b||^2
    int32_t iters, failed;
};

struct Ctx {
    int op = STA_OP_ELASTICITY;
    int64_t n = 0, T = 0, nblocks = 0, nnz = 0, nrows = 0;
    double eps = 0.0;
    int blocks_per_sm = 0;
    int rebuild_form = STA_REBUILD_AUTO;  // sta_set_rebuild_form
    int64_t n_active = 0;                 // active tetrahedra (host mirror count)
    int num_sms = 0;
    bool small_frames = false;    // the device runs k_frame_small
    int device = 0;

    // inputs
    double4_32a *X = nullptr;   // n, (x, y, z, 0)
    int4 *tets = nullptr;   // T
    double2 *mat = nullptr; // T, (E, nu)

    // pattern
    int32_t *adj_ptr = nullptr;    // n + 1: first block of node a
    int32_t *adj = nullptr;        // nblocks: neighbour node of each block (ascending per node)
    int32_t *block_node = nullptr; // nblocks: owner node of each block
    int32_t *row_ptr = nullptr;    // 3n + 1
    int32_t *col = nullptr;        // nnz
    int32_t *tblk = nullptr;       // T x 16: block of local pair (la, lb) = 4 la + lb
    int32_t *scat = nullptr;       // T x 144: CSR index of local entry (p, q)
    int2 *boff = nullptr;          // nblocks: {first value index, row stride}
    // Fold units: unordered node pairs {a <= b}.  Entry (3a+i, 3b+j) and its mirror
    // (3b+j, 3a+i) fold the same operands in the same order (the element matrices are exactly
    // symmetric), so one fold per unit writes both blocks.
    int64_t nunits = 0;
    int64_t nchunks = 0;
    int2 *chunks = nullptr;        // nchunks: rebuild fold chunks {first unit, units | diagonal << 8}
    uint8_t *cflag = nullptr;      // nchunks: the zero-fill rebuild's "fold this chunk"
    unsigned int *d_fault = nullptr;  // host-mapped word: a fold's bounded wait ran out
    unsigned int *h_fault = nullptr;
    bool fault_told = false;          // a call has reported it
    int4 *bmeta = nullptr;         // nunits: {value offset of (a,b), rs_a << 1 | diagonal, offset of
                                   //   the unit's first run, contributors}
    int2 *bmirror = nullptr;       // nunits: {value offset of (b,a), rs_b}
    UnitState *ustate = nullptr;   // nunits: contributor activity and claims
    uint32_t *uext = nullptr;      // activity words of contributors 64 and up
    int32_t *uc0 = nullptr;        // nunits + 1: first position of each unit's contributors in ctet
    int32_t *ctet = nullptr;       // 10 T: contributors of every unit, ascending tet id
    int32_t *tpos = nullptr;       // T x 10: tet t's place among the contributors of its slot's unit
    int32_t *krun = nullptr;       // T x 10: offset of tet t's run of a slot in Ke
    int32_t *tunit = nullptr;      // T x 10: unit of tet t's slot (4 diagonal, 6 pairs)
    int32_t *nt_ptr = nullptr;     // n + 1: node -> incident tetrahedra
    int32_t *nt_list = nullptr;    // 4 T: incident tetrahedra, ascending id
    uint8_t *steep = nullptr;      // T: local node whose barycentric gradient is about the largest (adjoint)
    double *dXe = nullptr;         // T x 12: per-element position gradients (adjoint, lazily)
    double *gunit = nullptr;       // nunits x 10: parts of each unit's gradient (adjoint, lazily)
    int32_t *nt_run = nullptr;     // 4 T: offset in dXe of each nt_list entry (adjoint, lazily)
    int32_t *act_list = nullptr;   // T: active tets, unordered (element / adjoint kernels, lazily)
    unsigned long long *act_count = nullptr;

    // state
    int64_t ke_len = 0;         // doubles of the element cache (<= 84 T)
    double *Ke = nullptr;       // ke_len: element cache
    // update policy (STA_POLICY_*) and the fixed-point state (sta_fixed.cu), allocated on first use
    int policy = STA_POLICY_REFOLD;
    long long *fx_q = nullptr;  // ke_len: quantised contributions at the element-cache offsets
    int16_t *fx_e = nullptr;    // nnz: exponent of each entry (keyed by its upper-block index)
    long long *fx_s = nullptr;  // nnz: exact integer sum of each entry's active contributions
    uint8_t *mask = nullptr;    // T
    double *val = nullptr;      // nnz
    int32_t *touched = nullptr; // nunits: list of units touched by the current frame
    // [0] bad elements, [1] touched units, [2] first bad element, [3] touched CSR entries
    unsigned long long *counters = nullptr;

    // streaming staging outside graph mode: two host-mapped pinned blocks used in turn, which the
    // kernels read where they are, each with an event of its last frame's end; and two sets of
    // device counters (each frame's last kernel zeroes the other set)
    // (one allocation, the first block's)
    FrameHeader *h_frame[2] = {nullptr, nullptr}, *m_frame[2] = {nullptr, nullptr};
    cudaEvent_t f_done[2] = {nullptr, nullptr};
    bool f_pending[2] = {false, false};
    int f_next = 0;
    unsigned long long *f_cnt = nullptr;  // 2 x 4
    int64_t edit_cap = 0;         // edited tetrahedra a frame block holds
    int64_t last_edited = 0;
    unsigned long long *last_counters = nullptr;  // device counters of the last frame
    // host-mapped pinned word the re-fold streaming frame's fold kernel stores its touched-entry
    // count into (h: host address, d: its device address); count_on_host: the last frame did
    unsigned long long *h_count_mapped = nullptr, *d_count_mapped = nullptr;
    bool count_on_host = false;
    uint8_t stamp_gen = 0;        // the sta_apply_edits call's stamp (1 .. 127), see tstate

    // graph-Laplacian proxy operator (sta_proxy.cu); its CSR is the node-level pattern
    // (row_ptr = adj_ptr, col = adj, nrows = n, nnz = nblocks)
    int32_t *ptblk = nullptr;   // T x 10: block of tet t's unit slot s (diagonal; upper edge block)
    int32_t *pmir = nullptr;    // nblocks: block (b, a) of block (a, b)
    int32_t *pup = nullptr;     // nblocks: upper block of the block's edge, -1 on the diagonal
    int32_t *pdiag = nullptr;   // n: diagonal block of each node, -1 for a node of no tetrahedron
    int32_t *pmult = nullptr;   // nblocks + n: edge multiplicity at the upper block, then degrees
    uint32_t *pflag = nullptr;  // nblocks: claim flags of the frame's touched blocks
    int32_t *plist = nullptr;   // nblocks: the frame's touched blocks

    // implicit-Euler loop (sta_dyn.cu), allocated by the first sta_dyn_setup
    bool dyn = false;
    double dyn_rho = 0.0, dyn_h = 0.0;
    double *qmass = nullptr;    // T: (rho V) / 4 of each tetrahedron
    double *mass = nullptr;     // n: lumped mass per node, maintained with the mask
    double *du = nullptr, *dv = nullptr, *df = nullptr;  // 3n: displacement, velocity, load
    uint8_t *clamped = nullptr; // n
    int32_t *dyn_perm = nullptr;  // n: sta_dyn_apply's node order (ascending row length)

    // conjugate gradients (sta_cg.cu), allocated by the first sta_dyn_setup or sta_solve
    double *cg = nullptr;       // x, b, D^-1 (nrows each), z (4 doubles a node of 3 DOFs, else 1)
    uint8_t *cg_free = nullptr; // nrows: DOF solved for
    int32_t *cg_snode = nullptr, *cg_sbase = nullptr, *cg_cta = nullptr, *cg_col = nullptr;  // slice plan
    double *cg_val = nullptr;   // the matrix of a solve in slice order
    double *cg_vec = nullptr;   // vectors in slice order when shared memory does not hold them
    void *cg_slots = nullptr;   // words of the grid-wide sums
    unsigned long long cg_epoch = 0;  // number of the last grid-wide sum given out
    unsigned cg_spins = 1u << 22;     // polls of a grid-wide wait at most (seconds)
    int cg_grid = 0, cg_S = 1, cg_warps = 1;
    int64_t cg_slices = 0, cg_steps = 0;
    bool cg_resident = false;   // shared memory keeps the matrix,
    bool cg_plan_shared = false;  // the nodes and steps of the slices
    size_t cg_smem = 0;
    CgResult *h_cg = nullptr, *d_cg = nullptr;  // host-mapped: a solve's result

    // CUDA-graph mode (sta_graph_enable): captured frame sequences and fixed staging
    bool graph_on = false;
    cudaGraphExec_t g_refold = nullptr, g_rebuild = nullptr;
    // graph mode stages frames in two host-mapped pinned blocks that the captured kernels read
    // directly (no copy call per frame), used alternately; each has its own captured sequence,
    // its own device counters (zeroed by the other sequence's last kernel) and an event
    // recorded after its launch, waited on before the block is written again
    int64_t gcap = 0;
    cudaGraphExec_t g_streams[2] = {nullptr, nullptr};
    FrameHeader *h_gframe[2] = {nullptr, nullptr};  // host-mapped pinned, gcap entries each
    FrameHeader *m_gframe[2] = {nullptr, nullptr};  // their device addresses
    unsigned long long *d_gcnt = nullptr;           // 2 x 4 counters
    cudaEvent_t g_done[2] = {nullptr, nullptr};
    bool g_pending[2] = {false, false};
    int g_next = 0;

    // batched form (sta_batch_create): instance offsets and per-instance CSR index arrays
    int32_t n_inst = 0;
    std::vector<int64_t> node_off, tet_off, nnz_off;
    int32_t *local_rp = nullptr;   // sum_i (3 n_i + 1): instance i at 3 node_off[i] + i
    int32_t *local_col = nullptr;  // nnz: column minus the instance's first DOF

    // host mirror of every tetrahedron, one byte: bit 7 = active (the mask), bits 0..6 = the
    // stamp of the last sta_apply_edits call that named it (duplicate check); one random
    // access per edited tetrahedron serves both checks
    std::vector<uint8_t> tstate;
    std::vector<uint8_t> seen;  // per-tet scratch for edit validation (all zero at rest)
    int64_t device_bytes = 0;
    std::vector<void *> allocations;
};

constexpr uint8_t TS_ACTIVE = 0x80;
constexpr uint8_t TS_STAMP = 0x7f;
inline bool ts_active(const Ctx *c, int64_t t) { return (c->tstate[t] & TS_ACTIVE) != 0; }
inline void ts_set_active(Ctx *c, int64_t t, bool on) {
    c->tstate[t] = (uint8_t)((c->tstate[t] & TS_STAMP) | (on ? TS_ACTIVE : 0));
}

// Launch of a kernel that may start while the stream's kernel before it still runs: it orders itself
// with dependency_wait(), before which it reads only what no kernel writes.  What the kernel before
// writes it reads after that with plain loads or from L2 (__ldcg), never over the read-only path
// (__ldg, const __restrict__), which asks that memory stays as it is from the kernel's start.
template <typename... P, typename... Q>
int launch_overlapped(void (*kern)(P...), unsigned grid, unsigned threads, size_t smem, cudaStream_t s,
                      Q... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    STA_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, P(args)...));
    return STA_OK;
}
#ifdef __CUDACC__
// the CTA has done what the kernel's successor has to wait for but for its end
__device__ __forceinline__ void launch_dependents() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// every kernel before this one in its stream is complete, its writes visible
__device__ __forceinline__ void dependency_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
#endif

template <typename T> int dev_alloc(Ctx *c, T **p, int64_t count) {
    size_t bytes = sizeof(T) * (size_t)(count > 0 ? count : 1);
    cudaError_t e = cudaMalloc((void **)p, bytes);
    if (e != cudaSuccess) {
        *p = nullptr;
        return fail(STA_ENOMEM, std::string("cudaMalloc failed: ") + cudaGetErrorString(e));
    }
    c->allocations.push_back((void *)*p);
    c->device_bytes += (int64_t)bytes;
    return STA_OK;
}

// Persistent grid for an item count: min(ceil(items / threads), SMs * CTAs per SM), CTAs per
// SM = the context's blocks_per_sm (the rebuild's tuned shape) if `tuned` and it is set, else
// the occupancy maximum.
int persistent_grid(const Ctx *c, const void *kernel, int threads, int64_t items,
                    bool tuned = false);

// ------------------------------------------------------------------------------------
// Kernel launchers (each returns STA_OK or STA_ECUDA on a launch error)
// ------------------------------------------------------------------------------------
int build_pattern(Ctx *c, cudaStream_t s);                       // sta_create.cu
int launch_elements(Ctx *c, bool active_only, cudaStream_t s);   // sta_element.cu
int launch_pack_params(Ctx *c, const double *nodes, const double *young, const double *poisson,
                       cudaStream_t s);
int launch_expand_elements(Ctx *c, const int32_t *ids, int64_t n, double *out, cudaStream_t s);
int launch_active_list(Ctx *c, double *dE, double *dnu, double *dXe, cudaStream_t s);
int launch_adjoint(Ctx *c, const double *gval, double *dE, double *dnu, double *dX, cudaStream_t s);  // sta_adjoint.cu
int launch_spmv(Ctx *c, const double *val, const double *x, double *y, cudaStream_t s);
int launch_rebuild(Ctx *c, cudaStream_t s);                      // sta_rebuild.cu
int rebuild_form_of(const Ctx *c);  // the form the next rebuild takes (AUTO resolved)
// Frames of at most this many edited tetrahedra take one launch, k_frame_small (elasticity, re-fold
// policy, without the dynamics' mass update).  The cluster's 112 warps fold the units of 40 tetrahedra
// that share none, 160 diagonal and 240 pair units, in one round each.  Two kernels take 8.3-8.9 us a
// frame back to back from 16 edits to 122, one cluster 5.6 us for 16, 5.8 for 32, 7.2 for 48, 7.4 for 60
// and 9.2 for 90; a frame that is waited for is even at 32 edits and 1.5 us longer at 48 (21.5 us).
constexpr int SMALL_FRAME = 40;
// In graph mode, frames of at most this many edited tetrahedra are launched kernel by kernel all the
// same.  Such a frame's kernels start as soon as the last CTA of the kernel before has left, without a
// graph's entry and exit, but its second launch costs host time, and back to back it takes what its
// call takes.  us a frame, graph / direct (two runs), on a block of 384,000 tetrahedra: edits in a plane,
// 600: 12.2 / 9.9-11.9, 1,000: 12.8 / 10.7-12.5, 1,500: 13.0 / 11.7-13.4, 2,000: 13.6 / 12.4-14.3,
// 3,000: 13.7 / 14.3-15.5; scattered, 600: 12.9 / 10.1-11.9, 2,000: 17.1 / 13.3-13.7, 4,000: 21.2 /
// 17.4.  So up to about 1,000 edits direct launches are the faster ones for both; above, only where
// the edits are scattered (the graph's kernels then take longer than the call), which the count does not
// tell.  A frame that is waited for takes as long either way, or up to 2 us less from the graph.
constexpr int DIRECT_FRAME = 1024;
int launch_small_frame(Ctx *c, const int32_t *edited, int m, bool replay, cudaStream_t s);
bool small_frames_fit();
// whether a streaming frame of this context stores its touched count into h_count_mapped
bool frame_counts_to_host(const Ctx *c);
// one streaming frame: the edited list, its count (*m_dev, or m) and the counters; cap: edited
// tetrahedra the grids are sized for; next_cnt: the counters the frame's last kernel zeroes for the
// next frame, or nullptr; replay: the caller captures the frame, and may replay it as it is
int launch_stream_frame(Ctx *c, const int32_t *edited, int64_t m, const int64_t *m_dev,
                        unsigned long long *cnt, int64_t cap, cudaStream_t s,
                        unsigned long long *next_cnt, bool replay);  // sta_stream.cu
bool capturing(cudaStream_t s);  // whether the stream records a CUDA graph of the caller's
int launch_fx_prepare(Ctx *c, cudaStream_t s);                   // sta_fixed.cu
int launch_fx_frame(Ctx *c, const int32_t *edited, int64_t m, const int64_t *m_dev, int64_t cap,
                    int32_t *touched, unsigned long long *counters, cudaStream_t s,
                    unsigned long long *next_cnt, bool replay);
int launch_mask_bits(Ctx *c, cudaStream_t s);                    // activity bits <- mask
int launch_values(Ctx *c, cudaStream_t s);  // the operator's rebuild (elasticity or proxy)
int launch_dyn_qmass(Ctx *c, cudaStream_t s);     // sta_dyn.cu (no-ops unless set up)
int launch_dyn_mass_all(Ctx *c, cudaStream_t s);
int launch_dyn_mass_edited(Ctx *c, const int32_t *edited, int64_t m, const int64_t *m_dev,
                           int64_t cap, cudaStream_t s);
int cg_alloc(Ctx *c);                              // sta_cg.cu
int launch_cg_solve(Ctx *c, const double *val, const double *mass, double h2, double tol,
                    int32_t max_iter, bool stagnate, double *xout, cudaStream_t s,
                    CgResult *res);
int build_proxy_maps(Ctx *c, const int32_t *tblk, cudaStream_t s);  // sta_proxy.cu
int launch_proxy_rebuild(Ctx *c, cudaStream_t s);
int launch_proxy_frame(Ctx *c, const int32_t *edited, int64_t m, const int64_t *m_dev,
                       int64_t cap, int32_t *list, unsigned long long *counters, cudaStream_t s,
                       unsigned long long *next_cnt);
int launch_stream_scratch(Ctx *c, int64_t m, const int32_t *d_edited, int32_t *touched,
                          unsigned long long *counters, cudaStream_t s);

int create_impl(const double *nodes, int64_t n_nodes, const int32_t *tets, int64_t n_tets,
                const double *young, const double *poisson, const sta_options *opt, void *stream,
                sta_ctx **out);
int check_values(Ctx *c);    // sta_api.cu: STA_ECUDA while the values are a failed rebuild's
void graph_release(Ctx *c);  // sta_graph.cu
int apply_frame(sta_ctx *x, const sta_edit *edits, int64_t n_edits, const int64_t *counts,
                void *stream);  // sta_api.cu

}  // namespace sta

// The opaque handle of the C-ABI.
struct sta_ctx {
    sta::Ctx c;
    cudaEvent_t h2d_done = nullptr;
    bool h2d_pending = false;
    uint8_t *h_mask = nullptr;  // pinned staging for host masks, T bytes
    unsigned long long *h_count = nullptr;  // 4 pinned words: read-back of device counters
};
