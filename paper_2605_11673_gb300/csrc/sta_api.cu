// C-ABI entry points of libsta (declared in include/sta.h): argument and edit validation on
// the host, device memory management, and the launch sequence of each call.
#include <algorithm>
#include <atomic>
#include <climits>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "sta_internal.cuh"

namespace sta {

static thread_local std::string g_last_error;

void set_error(const std::string &msg) { g_last_error = msg; }
int fail(int code, const std::string &msg) {
    set_error(msg);
    return code;
}

}  // namespace sta

using namespace sta;


// The host mirror of a new mask and its 0/1 staging copy; returns the active count.  Blocks of 128
// bytes whose count fits a byte: the compiler keeps every quantity in byte lanes (with a 64-bit
// count in the loop it widened every byte eight times: 202 us for 577,000 tetrahedra, this 27 us).
static int64_t set_host_mask(Ctx *c, const uint8_t *__restrict__ mask, uint8_t *__restrict__ stage) {
    uint8_t *__restrict__ ts = c->tstate.data();
    const int64_t T = c->T;
    int64_t na = 0, t = 0;
    for (; t + 128 <= T; t += 128) {
        uint8_t n = 0;
        for (int i = 0; i < 128; ++i) {
            const uint8_t on = mask[t + i] ? 1 : 0;
            ts[t + i] = (uint8_t)((ts[t + i] & TS_STAMP) | (on << 7));
            stage[t + i] = on;
            n = (uint8_t)(n + on);
        }
        na += n;
    }
    for (; t < T; ++t) {
        const uint8_t on = mask[t] ? 1 : 0;
        ts[t] = (uint8_t)((ts[t] & TS_STAMP) | (on << 7));
        stage[t] = on;
        na += on;
    }
    return na;
}

// Whether a bounded wait of an earlier rebuild ran out, which leaves its values incomplete.
static bool rebuild_failed(const Ctx *c) {
    return c->h_fault && *reinterpret_cast<volatile unsigned int *>(c->h_fault);
}

// For every call that reads or maintains the values.
int sta::check_values(Ctx *c) {
    if (!rebuild_failed(c)) return STA_OK;
    c->fault_told = true;
    return fail(STA_ECUDA, "an earlier rebuild did not complete: its values are incomplete until the next rebuild");
}

// For a rebuild: it reports an earlier one's failure that no call has reported yet, else puts it right.
static int begin_rebuild(Ctx *c, cudaStream_t s) {
    if (!rebuild_failed(c)) return STA_OK;
    if (!c->fault_told) return check_values(c);
    STA_CUDA_TRY(cudaStreamSynchronize(s));  // (the failed one may still be running)
    *reinterpret_cast<volatile unsigned int *>(c->h_fault) = 0u;
    c->fault_told = false;
    return STA_OK;
}

static int wait_staging(sta_ctx *x) {
    if (x->h2d_pending) {
        STA_CUDA_TRY(cudaEventSynchronize(x->h2d_done));
        x->h2d_pending = false;
    }
    return STA_OK;
}

static void free_ctx(sta_ctx *x) {
    if (!x) return;
    for (void *p : x->c.allocations) cudaFree(p);
    x->c.allocations.clear();
    if (x->c.h_frame[0]) cudaFreeHost(x->c.h_frame[0]);
    for (cudaEvent_t e : x->c.f_done)
        if (e) cudaEventDestroy(e);
    if (x->h_mask) cudaFreeHost(x->h_mask);
    if (x->h_count) cudaFreeHost(x->h_count);
    if (x->c.h_count_mapped) cudaFreeHost(x->c.h_count_mapped);
    if (x->c.h_fault) cudaFreeHost(x->c.h_fault);
    if (x->h2d_done) cudaEventDestroy(x->h2d_done);
    if (x->c.h_cg) cudaFreeHost(x->c.h_cg);
    graph_release(&x->c);
    delete x;
}

extern "C" {

void sta_default_options(sta_options *opt) {
    if (!opt) return;
    opt->eps = 0.0;
    opt->block_threads = 0;
    opt->blocks_per_sm = 0;
}

const char *sta_last_error(void) { return g_last_error.c_str(); }

const char *sta_status_string(int status) {
    switch (status) {
    case STA_OK: return "ok";
    case STA_EINVAL: return "invalid argument";
    case STA_ESTATE: return "invalid state";
    case STA_ERANGE: return "index range overflow";
    case STA_ENOMEM: return "out of memory";
    case STA_ECUDA: return "CUDA error";
    default: return "unknown status";
    }
}

int sta_create(const double *nodes, int64_t n_nodes, const int32_t *tets, int64_t n_tets,
               const double *young, const double *poisson, const sta_options *opt,
               void *stream, sta_ctx **out) {
    return sta::create_impl(nodes, n_nodes, tets, n_tets, young, poisson, opt, stream, out);
}

}  // extern "C"

int sta::create_impl(const double *nodes, int64_t n_nodes, const int32_t *tets, int64_t n_tets,
                     const double *young, const double *poisson, const sta_options *opt,
                     void *stream, sta_ctx **out) {
    if (!out) return fail(STA_EINVAL, "out is NULL");
    *out = nullptr;
    if (n_nodes < 0 || n_tets < 0) return fail(STA_EINVAL, "negative size");
    if ((n_nodes > 0 && !nodes) || (n_tets > 0 && (!tets || !young || !poisson)))
        return fail(STA_EINVAL, "NULL input array");
    if (n_tets >= (1LL << 27)) return fail(STA_ERANGE, "n_tets must be < 2^27");
    if (n_tets * KE_STRIDE >= (1LL << 31))  // element cache offsets of the folds are 31-bit
        return fail(STA_ERANGE, "n_tets must be < 2^31 / " + std::to_string(KE_STRIDE));
    if (3 * n_nodes + 1 > INT32_MAX) return fail(STA_ERANGE, "3 * n_nodes + 1 exceeds int32");
    for (int64_t t = 0; t < n_tets; ++t) {
        const int32_t *q = tets + 4 * t;
        for (int a = 0; a < 4; ++a) {
            if (q[a] < 0 || q[a] >= n_nodes)
                return fail(STA_EINVAL, "tet " + std::to_string(t) + ": node id out of range");
            for (int b = 0; b < a; ++b)
                if (q[a] == q[b])
                    return fail(STA_EINVAL, "tet " + std::to_string(t) + ": repeated node");
        }
    }
    sta_options o;
    sta_default_options(&o);
    if (opt) o = *opt;
    if (o.block_threads != 0 && o.block_threads != 64 && o.block_threads != 128 && o.block_threads != 256)
        return fail(STA_EINVAL, "block_threads must be 64, 128 or 256");
    if (o.blocks_per_sm < 0) return fail(STA_EINVAL, "blocks_per_sm must be >= 0");

    cudaStream_t s = (cudaStream_t)stream;
    sta_ctx *x = new sta_ctx();
    Ctx *c = &x->c;
    c->n = n_nodes;
    c->T = n_tets;
    c->eps = o.eps;
    c->blocks_per_sm = o.blocks_per_sm;
    int rc = STA_OK;
    auto bail = [&](int code) {
        free_ctx(x);
        return code;
    };
    if (cudaGetDevice(&c->device) != cudaSuccess ||
        cudaDeviceGetAttribute(&c->num_sms, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess)
        return bail(fail(STA_ECUDA, "no CUDA device"));
    c->small_frames = small_frames_fit();
    if (cudaEventCreateWithFlags(&x->h2d_done, cudaEventDisableTiming) != cudaSuccess)
        return bail(fail(STA_ECUDA, "cudaEventCreate failed"));

    // inputs: nodes padded to double4_32a, tets as int4, materials as double2
    std::vector<double> X4(4 * (size_t)(n_nodes > 0 ? n_nodes : 1), 0.0);
    for (int64_t v = 0; v < n_nodes; ++v)
        for (int k = 0; k < 3; ++k) X4[4 * v + k] = nodes[3 * v + k];
    std::vector<double> M2(2 * (size_t)(n_tets > 0 ? n_tets : 1), 0.0);
    for (int64_t t = 0; t < n_tets; ++t) {
        M2[2 * t] = young[t];
        M2[2 * t + 1] = poisson[t];
    }
    if ((rc = dev_alloc(c, &c->X, n_nodes)) || (rc = dev_alloc(c, &c->tets, n_tets)) ||
        (rc = dev_alloc(c, &c->mat, n_tets)) || (rc = dev_alloc(c, &c->counters, 4)))
        return bail(rc);
    if (cudaMemcpyAsync(c->X, X4.data(), sizeof(double4_32a) * n_nodes, cudaMemcpyHostToDevice, s) ||
        cudaMemcpyAsync(c->tets, tets, sizeof(int4) * n_tets, cudaMemcpyHostToDevice, s) ||
        cudaMemcpyAsync(c->mat, M2.data(), sizeof(double2) * n_tets, cudaMemcpyHostToDevice, s))
        return bail(fail(STA_ECUDA, "input copy failed"));

    if ((rc = build_pattern(c, s))) return bail(rc);

    if ((rc = dev_alloc(c, &c->Ke, c->ke_len)) || (rc = dev_alloc(c, &c->mask, n_tets)) ||
        (rc = dev_alloc(c, &c->val, c->nnz)) || (rc = dev_alloc(c, &c->steep, n_tets)))
        return bail(rc);
    unsigned long long init[4] = {0ull, 0ull, ~0ull, 0ull};
    if (cudaMemcpyAsync(c->counters, init, sizeof init, cudaMemcpyHostToDevice, s) ||
        cudaMemsetAsync(c->mask, 0, (size_t)(n_tets > 0 ? n_tets : 1), s) ||
        cudaMemsetAsync(c->val, 0, sizeof(double) * (size_t)(c->nnz > 0 ? c->nnz : 1), s))
        return bail(fail(STA_ECUDA, "init failed"));
    if ((rc = launch_elements(c, false, s))) return bail(rc);
    unsigned long long back[4];
    if (cudaMemcpyAsync(back, c->counters, sizeof back, cudaMemcpyDeviceToHost, s) ||
        cudaStreamSynchronize(s))
        return bail(fail(STA_ECUDA, std::string("element kernel failed: ") +
                                        cudaGetErrorString(cudaGetLastError())));
    if (back[0] != 0)
        return bail(fail(STA_EINVAL, std::to_string(back[0]) +
                                         " tetrahedra have det <= 0 (first: tet " +
                                         std::to_string(back[2]) + ")"));
    c->tstate.assign((size_t)n_tets, 0);
    c->seen.assign((size_t)n_tets, 0);
    c->last_counters = c->counters;
    if (cudaMallocHost((void **)&x->h_count, 4 * sizeof(unsigned long long)) != cudaSuccess ||
        cudaMallocHost((void **)&x->h_mask, (size_t)(n_tets > 0 ? n_tets : 1)) != cudaSuccess ||
        cudaHostAlloc((void **)&c->h_count_mapped, sizeof(unsigned long long),
                      cudaHostAllocMapped) != cudaSuccess ||
        cudaHostGetDevicePointer((void **)&c->d_count_mapped, c->h_count_mapped, 0) != cudaSuccess ||
        cudaHostAlloc((void **)&c->h_fault, sizeof(unsigned int), cudaHostAllocMapped) != cudaSuccess ||
        cudaHostGetDevicePointer((void **)&c->d_fault, c->h_fault, 0) != cudaSuccess)
        return bail(fail(STA_ENOMEM, "pinned host buffers"));
    *c->h_fault = 0u;
    *out = x;
    return STA_OK;
}

extern "C" int sta_proxy_create(int64_t n_nodes, const int32_t *tets, int64_t n_tets, double eps,
                                void *stream, sta_ctx **out) {
    if (!out) return fail(STA_EINVAL, "out is NULL");
    *out = nullptr;
    if (n_nodes < 0 || n_tets < 0) return fail(STA_EINVAL, "negative size");
    if (n_tets > 0 && !tets) return fail(STA_EINVAL, "NULL input array");
    if (n_tets >= (1LL << 27)) return fail(STA_ERANGE, "n_tets must be < 2^27");
    if (n_nodes + 1 > INT32_MAX) return fail(STA_ERANGE, "n_nodes + 1 exceeds int32");
    for (int64_t t = 0; t < n_tets; ++t) {
        const int32_t *q = tets + 4 * t;
        for (int a = 0; a < 4; ++a) {
            if (q[a] < 0 || q[a] >= n_nodes)
                return fail(STA_EINVAL, "tet " + std::to_string(t) + ": node id out of range");
            for (int b = 0; b < a; ++b)
                if (q[a] == q[b])
                    return fail(STA_EINVAL, "tet " + std::to_string(t) + ": repeated node");
        }
    }
    cudaStream_t s = (cudaStream_t)stream;
    sta_ctx *x = new sta_ctx();
    Ctx *c = &x->c;
    c->op = STA_OP_PROXY;
    c->policy = STA_POLICY_FIXED;  // the maintained-count update; REFOLD recounts touched entries
    c->n = n_nodes;
    c->T = n_tets;
    c->eps = eps;
    int rc = STA_OK;
    auto bail = [&](int code) {
        free_ctx(x);
        return code;
    };
    if (cudaGetDevice(&c->device) != cudaSuccess ||
        cudaDeviceGetAttribute(&c->num_sms, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess)
        return bail(fail(STA_ECUDA, "no CUDA device"));
    if (cudaEventCreateWithFlags(&x->h2d_done, cudaEventDisableTiming) != cudaSuccess)
        return bail(fail(STA_ECUDA, "cudaEventCreate failed"));
    if ((rc = dev_alloc(c, &c->tets, n_tets)) || (rc = dev_alloc(c, &c->counters, 4)))
        return bail(rc);
    if (cudaMemcpyAsync(c->tets, tets, sizeof(int4) * n_tets, cudaMemcpyHostToDevice, s))
        return bail(fail(STA_ECUDA, "input copy failed"));
    if ((rc = build_pattern(c, s))) return bail(rc);
    if ((rc = dev_alloc(c, &c->mask, n_tets)) || (rc = dev_alloc(c, &c->val, c->nnz))) return bail(rc);
    unsigned long long init[4] = {0ull, 0ull, ~0ull, 0ull};
    if (cudaMemcpyAsync(c->counters, init, sizeof init, cudaMemcpyHostToDevice, s) ||
        cudaMemsetAsync(c->mask, 0, (size_t)(n_tets > 0 ? n_tets : 1), s))
        return bail(fail(STA_ECUDA, "init failed"));
    if ((rc = launch_proxy_rebuild(c, s))) return bail(rc);  // all inactive: A = eps I
    if (cudaStreamSynchronize(s) != cudaSuccess)
        return bail(fail(STA_ECUDA, std::string("proxy create: ") +
                                        cudaGetErrorString(cudaGetLastError())));
    c->tstate.assign((size_t)n_tets, 0);
    c->seen.assign((size_t)n_tets, 0);
    c->last_counters = c->counters;
    if (cudaMallocHost((void **)&x->h_count, 4 * sizeof(unsigned long long)) != cudaSuccess ||
        cudaMallocHost((void **)&x->h_mask, (size_t)(n_tets > 0 ? n_tets : 1)) != cudaSuccess)
        return bail(fail(STA_ENOMEM, "pinned mask buffer"));
    *out = x;
    return STA_OK;
}

extern "C" {

int sta_destroy(sta_ctx *x) {
    if (!x) return STA_OK;
    cudaDeviceSynchronize();
    free_ctx(x);
    return STA_OK;
}

int sta_full_rebuild(sta_ctx *x, const uint8_t *mask, int mask_on_device, void *stream) {
    if (!x) return fail(STA_EINVAL, "ctx is NULL");
    Ctx *c = &x->c;
    if (c->T > 0 && !mask) return fail(STA_EINVAL, "mask is NULL");
    cudaStream_t s = (cudaStream_t)stream;
    STA_TRY(begin_rebuild(c, s));
    if (c->T > 0) {
        STA_TRY(wait_staging(x));
        if (mask_on_device) {  // read back for the host mirror; the device copy is the 0/1 one
            std::vector<uint8_t> hm((size_t)c->T);
            STA_CUDA_TRY(cudaMemcpyAsync(hm.data(), mask, (size_t)c->T, cudaMemcpyDeviceToHost, s));
            STA_CUDA_TRY(cudaStreamSynchronize(s));
            c->n_active = set_host_mask(c, hm.data(), x->h_mask);
        } else {
            c->n_active = set_host_mask(c, mask, x->h_mask);
        }
        STA_CUDA_TRY(cudaMemcpyAsync(c->mask, x->h_mask, (size_t)c->T, cudaMemcpyHostToDevice, s));
        STA_CUDA_TRY(cudaEventRecord(x->h2d_done, s));
        x->h2d_pending = true;
    }
    if (c->graph_on) {
        STA_CUDA_TRY(cudaGraphLaunch(c->g_rebuild, s));
        return STA_OK;
    }
    STA_TRY(launch_mask_bits(c, s));
    return launch_values(c, s);
}

int sta_set_launch(sta_ctx *x, int32_t block_threads, int32_t blocks_per_sm) {
    if (!x) return fail(STA_EINVAL, "ctx is NULL");
    if (block_threads != 0 && block_threads != 64 && block_threads != 128 && block_threads != 256)
        return fail(STA_EINVAL, "block_threads must be 0, 64, 128 or 256");
    if (blocks_per_sm < 0) return fail(STA_EINVAL, "blocks_per_sm must be >= 0");
    if (x->c.graph_on) return fail(STA_ESTATE, "disable graph mode before changing the launch shape");
    x->c.blocks_per_sm = blocks_per_sm;
    return STA_OK;
}

int sta_set_fold_depth(sta_ctx *x, int32_t operands_in_flight) {
    if (!x) return fail(STA_EINVAL, "ctx is NULL");
    if (operands_in_flight != 4 && operands_in_flight != 6)
        return fail(STA_EINVAL, "operands_in_flight must be 4 or 6");
    if (x->c.graph_on) return fail(STA_ESTATE, "disable graph mode before changing the fold depth");
    return STA_OK;
}

int sta_set_rebuild_form(sta_ctx *x, int32_t form) {
    if (!x) return fail(STA_EINVAL, "ctx is NULL");
    if (form != STA_REBUILD_AUTO && form != STA_REBUILD_FUSED && form != STA_REBUILD_ZERO_FILL)
        return fail(STA_EINVAL, "form must be STA_REBUILD_AUTO, _FUSED or _ZERO_FILL");
    if (x->c.graph_on) return fail(STA_ESTATE, "disable graph mode before changing the rebuild form");
    x->c.rebuild_form = form;
    return STA_OK;
}

int sta_get_rebuild_form(const sta_ctx *x, int32_t *form) {
    if (!x || !form) return fail(STA_EINVAL, "NULL argument");
    *form = rebuild_form_of(&x->c);
    return STA_OK;
}

int sta_refold(sta_ctx *x, void *stream) {
    if (!x) return fail(STA_EINVAL, "ctx is NULL");
    STA_TRY(begin_rebuild(&x->c, (cudaStream_t)stream));
    if (x->c.graph_on) {
        STA_CUDA_TRY(cudaGraphLaunch(x->c.g_refold, (cudaStream_t)stream));
        return STA_OK;
    }
    return launch_values(&x->c, (cudaStream_t)stream);
}

int sta_apply_edits(sta_ctx *x, const sta_edit *edits, int64_t n_edits, void *stream) {
    if (!x) return fail(STA_EINVAL, "ctx is NULL");
    if (n_edits < 0 || (n_edits > 0 && !edits)) return fail(STA_EINVAL, "bad edit list");
    return apply_frame(x, edits, n_edits, nullptr, stream);
}

}  // extern "C"

// Host-mapped frame blocks for `cap` edited tetrahedra each (the old ones are free once the frames
// that read them are done), and on first use their events and counters.
static int grow_frames(Ctx *c, int64_t cap, cudaStream_t s) {
    for (int b = 0; b < 2; ++b) {
        if (!c->f_done[b])
            STA_CUDA_TRY(cudaEventCreateWithFlags(&c->f_done[b], cudaEventDisableTiming));
        if (c->f_pending[b]) {
            STA_CUDA_TRY(cudaEventSynchronize(c->f_done[b]));
            c->f_pending[b] = false;
        }
    }
    if (!c->f_cnt) {
        STA_TRY(dev_alloc(c, &c->f_cnt, 8));
        STA_CUDA_TRY(cudaMemsetAsync(c->f_cnt, 0, 8 * sizeof(unsigned long long), s));
    }
    c->edit_cap = 0;
    if (c->h_frame[0]) cudaFreeHost(c->h_frame[0]);
    c->h_frame[0] = c->h_frame[1] = nullptr;
    const size_t stride = (frame_bytes(cap) + 127) & ~(size_t)127;
    char *h = nullptr;
    void *d = nullptr;
    if (cudaHostAlloc((void **)&h, 2 * stride, cudaHostAllocMapped) != cudaSuccess)
        return fail(STA_ENOMEM, "pinned edit buffer");
    c->h_frame[0] = reinterpret_cast<FrameHeader *>(h);
    c->h_frame[1] = reinterpret_cast<FrameHeader *>(h + stride);
    if (cudaHostGetDevicePointer(&d, h, 0) != cudaSuccess)
        return fail(STA_ENOMEM, "pinned edit buffer (host-mapped)");
    c->m_frame[0] = static_cast<FrameHeader *>(d);
    c->m_frame[1] = reinterpret_cast<FrameHeader *>(static_cast<char *>(d) + stride);
    c->edit_cap = cap;
    return STA_OK;
}

bool sta::capturing(cudaStream_t s) {  // (40 ns)
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &st) != cudaSuccess) cudaGetLastError();
    return st != cudaStreamCaptureStatusNone;
}

// What is wrong with an edit of tetrahedra [0, T) shifted by off, in the order of the checks.
static const char *edit_error(const Ctx *c, const sta_edit &E, int64_t T, int64_t off, uint8_t gen,
                              bool batch) {
    const char *range = batch ? "tet out of the instance's range" : nullptr;
    const uint8_t *ts = c->tstate.data() + off;
    if (batch && (E.tet < 0 || E.tet >= T || (E.op == STA_SWAP && (E.tet2 < 0 || E.tet2 >= T))))
        return range;
    if (E.op < 0 || E.op > 2) return "bad op";
    if (E.tet < 0 || E.tet >= T) return "tet out of range";
    const uint8_t s1 = ts[E.tet];
    if ((s1 & TS_STAMP) == gen) return "tet named twice";
    if (E.op == STA_DEACTIVATE) return s1 & TS_ACTIVE ? nullptr : "deactivating an inactive tet";
    if (E.op == STA_ACTIVATE) return s1 & TS_ACTIVE ? "activating an active tet" : nullptr;
    if (E.tet2 < 0 || E.tet2 >= T) return "tet2 out of range";
    const uint8_t s2 = ts[E.tet2];
    if (E.tet2 == E.tet || (s2 & TS_STAMP) == gen) return "tet2 named twice";
    if (!(s1 & TS_ACTIVE) || (s2 & TS_ACTIVE)) return "swap needs an active tet and an inactive tet2";
    return nullptr;
}

// One frame: `edits` in order, tet ids of the whole context, or with `counts` (batched context)
// counts[i] edits of instance i after one another with ids local to it.
int sta::apply_frame(sta_ctx *x, const sta_edit *edits, int64_t n_edits, const int64_t *counts,
                     void *stream) {
    Ctx *c = &x->c;
    if (n_edits > (INT32_MAX / 32)) return fail(STA_ERANGE, "too many edits in one call");
    STA_TRY(check_values(c));
    cudaStream_t s = (cudaStream_t)stream;
    // edited tetrahedra (a swap edits two): 2 n_edits bounds them; they are counted first only where
    // that bound is past the capacity of the block at hand, or the frame is a small one.  Staging
    // counts them exactly either way.
    int64_t m = 2 * n_edits;
    if (m > (c->graph_on ? c->gcap : c->edit_cap) || n_edits <= SMALL_FRAME) {
        m = n_edits;
        for (int64_t e = 0; e < n_edits; ++e) m += edits[e].op == STA_SWAP;
    }

    // the frame block to stage into: one of the graph mode's two host-mapped blocks (fixed
    // capacity), or the context's pinned block (grown on demand); a small frame needs neither
    const bool two_kernels = c->op == STA_OP_ELASTICITY && !c->dyn;
    const bool small = m > 0 && m <= SMALL_FRAME && two_kernels && c->policy == STA_POLICY_REFOLD &&
                       c->small_frames;
    const bool use_graph = c->graph_on && m <= c->gcap && !small;
    FrameHeader *h = nullptr, *d = nullptr;
    int32_t by_value[SMALL_FRAME];
    int gb = 0;
    if (small) {  // staged here: the edits go with the launch
    } else if (use_graph) {  // the staging block last used two frames ago: its kernels are done
        gb = c->g_next;
        if (c->g_pending[gb]) {
            STA_CUDA_TRY(cudaEventSynchronize(c->g_done[gb]));
            c->g_pending[gb] = false;
        }
        h = c->h_gframe[gb];
        d = c->m_gframe[gb];
    } else {
        gb = c->f_next;
        if (m > c->edit_cap || c->edit_cap == 0) {
            // (room for as many swaps: a frame of this size is not counted beforehand again)
            const int64_t cap = m < 1024 ? 1024 : std::max(m + m / 2, 2 * n_edits);
            STA_TRY(grow_frames(c, cap, s));
        }
        if (c->f_pending[gb]) {  // the block's last frame, two frames ago, has read it
            STA_CUDA_TRY(cudaEventSynchronize(c->f_done[gb]));
            c->f_pending[gb] = false;
        }
        h = c->h_frame[gb];
        d = c->m_frame[gb];
    }

    // one pass: validate each edit against the host mirror of the mask, stage it and apply it
    // to the mirror; on a bad edit, undo the mirror changes made so far and change nothing
    if (++c->stamp_gen > TS_STAMP) {  // stamps wrapped (every 127 calls): clear them
        for (auto &b : c->tstate) b &= TS_ACTIVE;
        c->stamp_gen = 1;
    }
    const uint8_t gen = c->stamp_gen;
    uint8_t *ts = c->tstate.data();
    int32_t *stage = small ? by_value : frame_edited(h);
    int64_t k = 0, e = 0, dact = 0;  // dact: change of the active count
    bool bad = false;
    // (ids compare as unsigned, and an edit's state tests are one condition: the order of the
    // checks matters only for the message, which edit_error finds again.  The kinds of edit keep
    // branches of their own: edits of a kind come in runs, and one branchless form for both cost a
    // frame of 40,000 deactivations 75 us instead of 65.)
    const int64_t segments = counts ? c->n_inst : 1;
    int64_t seg = 0, seg0 = 0;
    for (; seg < segments && !bad; seg += !bad) {
        const int64_t off = counts ? c->tet_off[seg] : 0;
        const uint64_t T = (uint64_t)(counts ? c->tet_off[seg + 1] - off : c->T);
        const int64_t end = counts ? e + counts[seg] : n_edits;
        uint8_t *st = ts + off;
        const uint32_t o32 = (uint32_t)off;
        seg0 = e;
        for (; e < end; ++e) {
            if (e + 16 < n_edits) {  // the per-tet state is accessed at random: fetch it ahead
                // (a prefetch never faults, so an unchecked id -- tet2 of a non-swap is -1 -- costs
                // at most a useless prefetch; the address is formed as an integer)
                const sta_edit &F = edits[e + 16];
                const uintptr_t base = (uintptr_t)st;
                __builtin_prefetch((const void *)(base + (uintptr_t)(intptr_t)F.tet), 1);
                __builtin_prefetch((const void *)(base + (uintptr_t)(intptr_t)F.tet2), 1);
            }
            const sta_edit &E = edits[e];
            const uint32_t a = (uint32_t)E.tet;
            if ((uint32_t)E.op > 2u || a >= T) { bad = true; break; }
            const uint8_t s1 = st[a];
            if (E.op == STA_SWAP) {
                const uint32_t b = (uint32_t)E.tet2;
                if (b >= T) { bad = true; break; }
                const uint8_t s2 = st[b];
                if (((s1 & TS_STAMP) == gen) | ((s2 & TS_STAMP) == gen) | (a == b) |
                    ((s1 & TS_ACTIVE) == 0) | ((s2 & TS_ACTIVE) != 0)) { bad = true; break; }
                st[a] = gen;
                st[b] = (uint8_t)(TS_ACTIVE | gen);
                stage[k] = (int32_t)(a + o32);
                stage[k + 1] = (int32_t)((b + o32) | 0x80000000u);
                k += 2;
            } else if (E.op == STA_DEACTIVATE) {
                if (((s1 & TS_STAMP) == gen) | ((s1 & TS_ACTIVE) == 0)) { bad = true; break; }
                st[a] = gen;
                stage[k++] = (int32_t)(a + o32);
                --dact;
            } else {
                if (((s1 & TS_STAMP) == gen) | ((s1 & TS_ACTIVE) != 0)) { bad = true; break; }
                st[a] = (uint8_t)(TS_ACTIVE | gen);
                stage[k++] = (int32_t)((a + o32) | 0x80000000u);
                ++dact;
            }
        }
    }
    if (bad) {
        const int64_t off = counts ? c->tet_off[seg] : 0;
        const char *why = edit_error(c, edits[e], counts ? c->tet_off[seg + 1] - off : c->T, off, gen,
                                     counts != nullptr);
        for (int64_t r = 0; r < k; ++r)  // undo (each tet appears once, so this is exact)
            ts_set_active(c, (uint32_t)stage[r] & 0x7fffffffu, stage[r] >= 0);
        return fail(STA_EINVAL, (counts ? "instance " + std::to_string(seg) + ", edit " +
                                              std::to_string(e - seg0)
                                        : "edit " + std::to_string(e)) +
                                    ": " + (why ? why : "rejected"));
    }
    c->n_active += dact;
    m = k;
    c->last_edited = m;
    if (small) {
        c->last_counters = c->counters;
        c->count_on_host = true;
        return launch_small_frame(c, stage, (int)m, capturing(s), s);
    }

    // the kernels read the host-mapped block itself: no copy call
    h->m = m;
    // the fold kernel stores the frame's touched count into the host-mapped word (a frame
    // without edits launches no kernel outside graph mode)
    c->count_on_host = frame_counts_to_host(c) && (use_graph || m > 0);
    std::atomic_thread_fence(std::memory_order_seq_cst);  // the block before the launch
    if (use_graph) {
        unsigned long long *cnt = c->d_gcnt + 4 * gb;
        c->last_counters = cnt;
        if (m > 0 && m <= DIRECT_FRAME && two_kernels && !capturing(s))
            STA_TRY(launch_stream_frame(c, frame_edited(d), m, nullptr, cnt, m, s,
                                        c->d_gcnt + 4 * (gb ^ 1), false));
        else
            STA_CUDA_TRY(cudaGraphLaunch(c->g_streams[gb], s));
        STA_CUDA_TRY(cudaEventRecord(c->g_done[gb], s));
        c->g_pending[gb] = true;
        c->g_next = gb ^ 1;
        return STA_OK;
    }
    if (m == 0) {
        c->last_counters = c->counters;
        STA_CUDA_TRY(cudaMemsetAsync(c->counters + 1, 0, 3 * sizeof(unsigned long long), s));
        return STA_OK;
    }
    unsigned long long *cnt = c->f_cnt + 4 * gb;
    c->last_counters = cnt;
    // (a captured frame may be replayed without the other block's frame, which zeroes these, in between)
    const bool replay = capturing(s);
    if (replay) STA_CUDA_TRY(cudaMemsetAsync(cnt, 0, 4 * sizeof(unsigned long long), s));
    STA_TRY(launch_stream_frame(c, frame_edited(d), m, nullptr, cnt, m, s, c->f_cnt + 4 * (gb ^ 1), replay));
    STA_CUDA_TRY(cudaEventRecord(c->f_done[gb], s));
    c->f_pending[gb] = true;
    c->f_next = gb ^ 1;
    return STA_OK;
}

extern "C" {

int sta_last_touched(sta_ctx *x, int64_t *touched_nnz, void *stream) {
    if (!x || !touched_nnz) return fail(STA_EINVAL, "NULL argument");
    STA_TRY(check_values(&x->c));
    cudaStream_t s = (cudaStream_t)stream;
    if (x->c.count_on_host) {  // the frame's fold kernel stored it in host-mapped memory
        STA_CUDA_TRY(cudaStreamSynchronize(s));
        STA_TRY(check_values(&x->c));
        *touched_nnz = (int64_t)*reinterpret_cast<volatile unsigned long long *>(x->c.h_count_mapped);
        return STA_OK;
    }
    // into a pinned word: a plain asynchronous copy (a pageable target is staged, and slower)
    STA_CUDA_TRY(cudaMemcpyAsync(x->h_count, x->c.last_counters + 3, sizeof *x->h_count,
                                 cudaMemcpyDeviceToHost, s));
    STA_CUDA_TRY(cudaStreamSynchronize(s));
    STA_TRY(check_values(&x->c));
    *touched_nnz = (int64_t)*x->h_count;
    return STA_OK;
}

int sta_csr(const sta_ctx *x, const int32_t **row_ptr, const int32_t **col, const double **val,
            int64_t *n_rows, int64_t *nnz) {
    if (!x) return fail(STA_EINVAL, "ctx is NULL");
    if (row_ptr) *row_ptr = x->c.row_ptr;
    if (col) *col = x->c.col;
    if (val) *val = x->c.val;
    if (n_rows) *n_rows = x->c.nrows;
    if (nnz) *nnz = x->c.nnz;
    return STA_OK;
}

int sta_scatter_map(const sta_ctx *x, const int32_t **scat) {
    if (!x || !scat) return fail(STA_EINVAL, "NULL argument");
    if (x->c.op != STA_OP_ELASTICITY) return fail(STA_ESTATE, "not an elasticity context");
    *scat = x->c.scat;
    return STA_OK;
}

int sta_mask(const sta_ctx *x, const uint8_t **mask) {
    if (!x || !mask) return fail(STA_EINVAL, "NULL argument");
    *mask = x->c.mask;
    return STA_OK;
}

int sta_sizes(const sta_ctx *x, int64_t *n_nodes, int64_t *n_tets, int64_t *n_blocks,
              int64_t *device_bytes) {
    if (!x) return fail(STA_EINVAL, "ctx is NULL");
    if (n_nodes) *n_nodes = x->c.n;
    if (n_tets) *n_tets = x->c.T;
    if (n_blocks) *n_blocks = x->c.nblocks;
    if (device_bytes) *device_bytes = x->c.device_bytes;
    return STA_OK;
}

int sta_recompute_elements(sta_ctx *x, int active_only, void *stream) {
    if (!x) return fail(STA_EINVAL, "ctx is NULL");
    if (x->c.op != STA_OP_ELASTICITY) return fail(STA_ESTATE, "not an elasticity context");
    STA_TRY(launch_elements(&x->c, active_only != 0, (cudaStream_t)stream));
    if (x->c.policy == STA_POLICY_FIXED) STA_TRY(launch_fx_prepare(&x->c, (cudaStream_t)stream));
    return STA_OK;
}

int sta_set_policy(sta_ctx *x, int32_t policy, void *stream) {
    if (!x) return fail(STA_EINVAL, "ctx is NULL");
    if (policy != STA_POLICY_REFOLD && policy != STA_POLICY_FIXED)
        return fail(STA_EINVAL, "policy must be STA_POLICY_REFOLD or STA_POLICY_FIXED");
    Ctx *c = &x->c;
    if (c->graph_on) return fail(STA_ESTATE, "disable graph mode before changing the policy");
    cudaStream_t s = (cudaStream_t)stream;
    STA_TRY(begin_rebuild(c, s));
    if (c->op == STA_OP_PROXY) {  // integer state either way: nothing to prepare
        c->policy = policy;
        return launch_values(c, s);
    }
    if (policy == STA_POLICY_FIXED) STA_TRY(launch_fx_prepare(c, s));
    c->policy = policy;
    return launch_rebuild(c, s);  // every value under the new policy, from the current mask
}

int sta_set_params(sta_ctx *x, const double *nodes, const double *young, const double *poisson,
                   int on_device, void *stream) {
    if (!x) return fail(STA_EINVAL, "ctx is NULL");
    if (x->c.op != STA_OP_ELASTICITY) return fail(STA_ESTATE, "not an elasticity context");
    Ctx *c = &x->c;
    cudaStream_t s = (cudaStream_t)stream;
    if (on_device) {
        STA_TRY(launch_pack_params(c, nodes, young, poisson, s));
    } else {
        if (nodes) {
            std::vector<double> X4(4 * (size_t)(c->n > 0 ? c->n : 1), 0.0);
            for (int64_t v = 0; v < c->n; ++v)
                for (int k = 0; k < 3; ++k) X4[4 * v + k] = nodes[3 * v + k];
            STA_CUDA_TRY(cudaMemcpyAsync(c->X, X4.data(), sizeof(double4_32a) * c->n,
                                         cudaMemcpyHostToDevice, s));
            STA_CUDA_TRY(cudaStreamSynchronize(s));
        }
        if (young)
            STA_CUDA_TRY(cudaMemcpy2DAsync(c->mat, sizeof(double2), young, sizeof(double),
                                           sizeof(double), (size_t)c->T, cudaMemcpyHostToDevice, s));
        if (poisson)
            STA_CUDA_TRY(cudaMemcpy2DAsync((double *)c->mat + 1, sizeof(double2), poisson,
                                           sizeof(double), sizeof(double), (size_t)c->T,
                                           cudaMemcpyHostToDevice, s));
        STA_TRY(launch_pack_params(c, nullptr, nullptr, nullptr, s));  // the counters
    }
    STA_TRY(launch_elements(c, false, s));
    unsigned long long *back = x->h_count;  // pinned: a pageable target is staged, and slower
    STA_CUDA_TRY(cudaMemcpyAsync(back, c->counters, 4 * sizeof *back, cudaMemcpyDeviceToHost, s));
    STA_CUDA_TRY(cudaStreamSynchronize(s));
    if (back[0] != 0)
        return fail(STA_EINVAL, std::to_string(back[0]) + " tetrahedra have det <= 0 (first: tet " +
                                    std::to_string(back[2]) + ")");
    if (c->policy == STA_POLICY_FIXED) STA_TRY(launch_fx_prepare(c, s));
    if (nodes) {  // the tetrahedra's volumes, hence the lumped mass, follow the positions
        STA_TRY(launch_dyn_qmass(c, s));
        STA_TRY(launch_dyn_mass_all(c, s));
    }
    return STA_OK;
}

int sta_adjoint(sta_ctx *x, const double *grad_val, double *dE, double *dnu, double *dX,
                void *stream) {
    if (!x) return fail(STA_EINVAL, "ctx is NULL");
    const Ctx *c = &x->c;
    if (x->c.op != STA_OP_ELASTICITY) return fail(STA_ESTATE, "not an elasticity context");
    if ((c->nnz > 0 && !grad_val) || (c->T > 0 && (!dE || !dnu)) || (c->n > 0 && !dX))
        return fail(STA_EINVAL, "NULL argument");
    return launch_adjoint(&x->c, grad_val, dE, dnu, dX, (cudaStream_t)stream);
}

int sta_spmv(sta_ctx *x, const double *val, const double *xv, double *y, void *stream) {
    if (!x) return fail(STA_EINVAL, "ctx is NULL");
    if (x->c.nrows > 0 && (!xv || !y)) return fail(STA_EINVAL, "NULL argument");
    STA_TRY(check_values(&x->c));
    return launch_spmv(&x->c, val ? val : x->c.val, xv, y, (cudaStream_t)stream);
}

int sta_element_matrices(sta_ctx *x, const int32_t *tet_ids, int64_t n, double *out, void *stream) {
    if (!x || n < 0 || (n > 0 && (!tet_ids || !out))) return fail(STA_EINVAL, "bad argument");
    if (x->c.op != STA_OP_ELASTICITY) return fail(STA_ESTATE, "not an elasticity context");
    return launch_expand_elements(&x->c, tet_ids, n, out, (cudaStream_t)stream);
}

}  // extern "C"
