// ivb_api.cu -- the C ABI declared in include/ivb.h: problem handles, input
// validation, the device node queue, the batched persistent launch replayed as
// a CUDA graph, the plain one-node-per-launch path, the autotuner, per-subdomain
// enclosures and point gradients.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>
#include <string>
#include <thread>
#include <vector>

#include "../../include/ivb.h"
#include "ivb_compile.h"
#include "ivb_internal.h"
#include "ivb_kernels.h"
#include "ivb_launch.h"
#include "ivb_problem.h"


using namespace ivb;


namespace {

thread_local std::string g_create_error;

ivb_status fail(ivb_problem* p, ivb_status st, const std::string& msg) {
    if (p) p->err = msg;
    else g_create_error = msg;
    return st;
}

ivb_status cuda_fail(ivb_problem* p, cudaError_t e, const char* where) {
    return fail(p, e == cudaErrorMemoryAllocation ? IVB_ENOMEM : IVB_ECUDA,
                std::string(where) + ": " + cudaGetErrorString(e));
}

#define CK(call)                                                  \
    do {                                                          \
        cudaError_t e_ = (call);                                  \
        if (e_ != cudaSuccess) return cuda_fail(p, e_, #call);    \
    } while (0)

bool is_device_ptr(const void* ptr) {
    if (!ptr) return false;
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, ptr) != cudaSuccess) { cudaGetLastError(); return false; }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

int kernel_mode(const ivb_problem* p, bool store) {
    const bool adj = p->opt.grad_mode == IVB_GRAD_ADJOINT;
    return store ? (adj ? KM_ADJ_STORE : KM_FWD_STORE) : (adj ? KM_ADJ_REDUCE : KM_FWD_REDUCE);
}

// per-thread frame of the tape interpreter (store modes, and the reduce mode
// when no tape-specialised kernel is loaded)
int frame_units(const ivb_problem* p) {
    return p->opt.grad_mode == IVB_GRAD_ADJOINT ? p->P.L.total_adj : p->P.L.total_fwd;
}

bool use_jit(const ivb_problem* p) { return p->jit.kern != nullptr; }

// the reduce launches run the tape-specialised kernel (loaded, and not
// outtimed by the interpreter in the autotuner)
bool reduce_jit(const ivb_problem* p) { return use_jit(p) && !p->tuned_interp; }

// per-thread units of device memory the reduce kernel needs: the interpreter's
// frame, a segmented kernel's state area, nothing for the other specialised
// kernels (registers only)
int reduce_units(const ivb_problem* p) {
    if (!reduce_jit(p)) return frame_units(p);
    return p->jit.state_units;
}

// staging of a call's small arrays goes through pinned memory (a pageable copy of a
// few bytes costs some 10 us of host time each); larger calls copy directly
constexpr size_t kPinnedMost = 1 << 20;

// Validate boxes and splits, write the node queue into the pinned staging
// buffer; returns the queue size in bytes through *bytes.
ivb_status stage_queue(ivb_problem* p, int n_nodes, const double* boxes, const int32_t* splits, long long g_begin,
                       long long g_count, bool enclose, size_t* bytes, long long* total_out, cudaStream_t s) {
    const int n = p->n;
    // host arrays are read in place; device arrays come over in two copies and one
    // wait (validation needs the values)
    const size_t bb = (size_t)n_nodes * n * 2 * sizeof(double), sb = (size_t)n_nodes * n * sizeof(int32_t);
    const bool db = is_device_ptr(boxes), ds = is_device_ptr(splits);
    std::vector<char> pageable;
    const double* B = boxes;
    const int32_t* S = splits;
    if (db || ds) {
        char* to = nullptr;
        if (bb + sb <= kPinnedMost) {
            const ivb_status st = ensure_pinned(p, p->h_in, bb + sb);
            if (st) return st;
            to = p->h_in.p;
        } else {
            pageable.resize(bb + sb);
            to = pageable.data();
        }
        if (db) { CK(cudaMemcpyAsync(to, boxes, bb, cudaMemcpyDeviceToHost, s)); B = reinterpret_cast<double*>(to); }
        if (ds) { CK(cudaMemcpyAsync(to + bb, splits, sb, cudaMemcpyDeviceToHost, s)); S = reinterpret_cast<int32_t*>(to + bb); }
        CK(cudaStreamSynchronize(s));
    }
    // the previous call's copy out of the staging buffer must have finished
    CK(cudaEventSynchronize(p->queue_free));
    char* q = p->h_queue;
    long long* hdr = reinterpret_cast<long long*>(q);
    long long* off = reinterpret_cast<long long*>(q + kQueueHeader);
    char* recs = q + kQueueHeader + 8 * (size_t)(n_nodes + 1);
    long long acc = 0;
    const double lim = std::ldexp(1.0, 1000);
    for (int nd = 0; nd < n_nodes; ++nd) {
        double* lo = reinterpret_cast<double*>(recs + (size_t)nd * p->rec_bytes);
        double* hi = lo + n;
        double* h = hi + n;
        int32_t* N = reinterpret_cast<int32_t*>(h + n);
        long long cnt = 1;
        for (int i = 0; i < n; ++i) {
            double ab[2];
            int32_t k;
            std::memcpy(ab, B + ((size_t)nd * n + i) * 2, sizeof ab);
            std::memcpy(&k, S + (size_t)nd * n + i, sizeof k);
            const double a = ab[0], b = ab[1];
            if (!std::isfinite(a) || !std::isfinite(b) || !(a <= b))
                return fail(p, IVB_EINVAL, "node " + std::to_string(nd) + ": box bounds must be finite with lo <= hi");
            if (std::fabs(a) > lim || std::fabs(b) > lim)
                return fail(p, IVB_EINVAL, "node " + std::to_string(nd) + ": |box endpoint| exceeds 2^1000");
            if (k < 1) return fail(p, IVB_EINVAL, "node " + std::to_string(nd) + ": splits must be >= 1");
            cnt *= k;
            if (cnt > (1LL << 31))
                return fail(p, IVB_EINVAL, "node " + std::to_string(nd) + ": product of splits exceeds 2^31");
            lo[i] = a;
            hi[i] = b;
            h[i] = (b - a) / (double)k;   // RN(RN(hi - lo) / N), as in the subdomain endpoint formula
            N[i] = k;
        }
        off[nd] = acc;
        acc += cnt;
    }
    off[n_nodes] = acc;
    long long g_end = acc;
    if (enclose) {
        if (g_begin < 0 || g_count < 0 || g_begin + g_count > acc)
            return fail(p, IVB_EINVAL, "subdomain range outside the node");
        g_end = g_begin + g_count;
    }
    hdr[0] = n_nodes;
    hdr[1] = g_end;
    *bytes = queue_bytes(n_nodes, n);
    *total_out = g_end;
    return IVB_OK;
}

void drop_graphs(ivb_problem* p) {
    for (cudaGraphExec_t& g : p->gexec)
        if (g) { cudaGraphExecDestroy(g); g = nullptr; }
}

void free_frame(ivb_problem* p) {
    if (p->d_frame) cudaFree(p->d_frame);
    p->d_frame = nullptr;
    p->frame_bytes = 0;
    drop_graphs(p);
}

// frames of `units` for a launch of exactly `grid` blocks
ivb_status ensure_frame(ivb_problem* p, int grid, int block, int units) {
    const size_t need = (size_t)grid * block * units * sizeof(double);
    if (need <= p->frame_bytes) return IVB_OK;
    free_frame(p);
    const cudaError_t e = cudaMalloc(&p->d_frame, need);
    if (e != cudaSuccess) {
        cudaGetLastError();   // the launches that follow check for it
        p->d_frame = nullptr;
        return cuda_fail(p, e, "frames");
    }
    p->frame_bytes = need;
    return IVB_OK;
}

// frames for a launch of at most *grid blocks; *grid becomes the number that the memory holds
ivb_status fit_frame(ivb_problem* p, int* grid, int block, int units) {
    const size_t per = (size_t)block * units * sizeof(double);
    if (per == 0) return IVB_OK;
    if ((size_t)*grid * per > p->frame_most) *grid = std::max(1, (int)(p->frame_most / per));
    ivb_status st = IVB_OK;
    const int got = blocks_that_fit(*grid, [&](int g) {
        st = ensure_frame(p, g, block, units);
        return st != IVB_ENOMEM;
    });
    if (st) return st;
    if (got < *grid) {
        p->frame_most = p->frame_bytes;   // not tried again on every call
        p->err.clear();
    }
    *grid = got;
    return IVB_OK;
}

KParams make_params(ivb_problem* p, int frame_smem) {
    KParams K{};
    K.prog = p->d_prog;
    K.queue = p->d_queue;
    K.rec_bytes = p->rec_bytes;
    K.counter = p->d_counter;
    K.tile = p->tile;
    K.gframe = p->d_frame;
    K.frame_in_smem = frame_smem;
    K.frame_units = reduce_units(p);
    K.keys = p->d_keys;
    K.form = p->opt.form;
    K.groups = 1;
    return K;
}

size_t smem_bytes(const ivb_problem* p, int block, int frame_smem) {
    return frame_smem ? (size_t)block * frame_units(p) * sizeof(double) : 0;
}

// the reduce-mode bounding kernel: tape-specialised when compiled, else the interpreter
cudaError_t launch_reduce(ivb_problem* p, KParams K, int grid, int block, int frame_smem, cudaStream_t s,
                          int tpsub, bool sync) {
    K.groups = tpsub;
    if (reduce_jit(p)) return jit_launch(p->jit, K, grid, block, s, tpsub, sync);
    return launch_bound(kernel_mode(p, false), K, grid, block, smem_bytes(p, block, frame_smem), s);
}

// resident blocks per SM of the reduce kernel
int reduce_occupancy(ivb_problem* p, int block, int frame_smem, int tpsub = 1, bool sync = false) {
    if (reduce_jit(p)) return block <= p->jit.max_threads ? jit_occupancy(p->jit, block, tpsub, sync) : 0;
    return occupancy_blocks(kernel_mode(p, false), block, smem_bytes(p, block, frame_smem));
}

// enqueue: keys, counter, bound kernel, finalize (the batched graph body)
ivb_status enqueue_bound(ivb_problem* p, int grid, int block, int tile, int frame_smem, int max_nodes, cudaStream_t s,
                         int tpsub, bool sync) {
    CK(launch_init_keys(p->d_keys, p->d_queue, max_nodes, p->n_out, p->d_counter, s));
    KParams K = make_params(p, frame_smem);
    K.tile = tile;
    CK(launch_reduce(p, K, grid, block, frame_smem, s, tpsub, sync));
    FinalizeParams F{};
    F.keys = p->d_keys;
    F.queue = p->d_queue;
    F.max_nodes = max_nodes;
    F.n_out = p->n_out;
    F.obj = p->obj;
    F.filter = p->opt.filter;
    F.out_kind = p->d_out_kind;
    F.out_in_header = true;
    CK(launch_finalize(F, s));
    p->launches += 3;
    return IVB_OK;
}

struct TuneCand {
    int block, bps, smem, tpsub, tile_mult;
    bool sync, interp;
};

// subdomains a block covers per pass of its tile loop
int pass_size(const ivb_problem* p, int block, int tpsub) {
    const int ilp = reduce_jit(p) && p->jit.state_units > 0 ? p->jit.ilp : 1;
    return block / std::max(1, tpsub) * ilp;
}

// threads-per-subdomain values the loaded kernel offers (1 unless segmented)
std::vector<int> tpsub_choices(const ivb_problem* p) {
    std::vector<int> v{1};
    if (reduce_jit(p))
        for (int t : {2, 4})
            if (p->jit.kern_t[tpsub_index(t)] && (p->opt.threads_per_subdomain == 0 || p->opt.threads_per_subdomain == t))
                v.push_back(t);
    if (p->opt.threads_per_subdomain > 1 && v.size() > 1) v.erase(v.begin());   // a fixed T > 1 excludes 1
    return v;
}

// Threads per subdomain of one call. A call whose subdomains do not fill the
// resident threads runs at the latency of its program, so the outputs of a
// subdomain are shared among as many threads as stay resident, unless an option
// fixes their number or the grabs (1024 subdomains of configuration 2, 4 outputs: 147 us with 1
// thread, 94 with 2, 76 with 4; the interpreter shares them among warp groups:
// 297 us with one group, 103 with 4).
int call_tpsub(const ivb_problem* p, long long total, long long threads) {
    if (p->opt.threads_per_subdomain != 0 || p->opt.tile > 0 || (reduce_jit(p) && p->jit.ilp != 1)) return p->tpsub;
    int best = p->tpsub;
    for (int t : {2, 4}) {
        const bool can = reduce_jit(p) ? p->jit.kern_t[tpsub_index(t)] != nullptr
                                       : p->opt.grad_mode == IVB_GRAD_ADJOINT && t <= p->n_out;
        if (t > best && can && groups_fit(p->block, t) && total * t <= threads) best = t;
    }
    return best;
}

// chunk synchronisation choices: the segmented kernels come with and without;
// programs larger than the instruction caches always keep their warps together
std::vector<bool> sync_choices(const ivb_problem* p) {
    if (!reduce_jit(p) || !p->jit.kern_sync[0]) return {false};
    if (p->opt.seg_sync == 0) return {false};
    if (p->opt.seg_sync == 1 || p->jit.chunks >= kSegSyncChunks) return {true};
    return {false, true};
}

ivb_status default_tuning(ivb_problem* p);

// Pick block size, blocks per SM, frame placement, threads per subdomain and
// subdomains per grab (tile) by timing the bound kernel on the first
// subdomains of the staged batch (results do not depend on the choice; a candidate
// whose frames do not fit is left out). The timed index range is capped at two
// waves of the widest candidate grid, and a candidate whose warm-up is already far
// slower than the best is not timed again, so that tuning stays a small fraction of a few calls. Stage 1 times every
// (threads per subdomain, block, blocks per SM, frame placement); stage 2
// times larger grabs (4 and 16 passes per grab) for the best of stage 1.
ivb_status autotune(ivb_problem* p, long long total, cudaStream_t s) {
    std::vector<TuneCand> cands;
    const int blocks[] = {1024, 512, 256, 128, 64};   // largest: segmented kernels 1024, interpreter 512
    const int bpss[] = {1, 2, 3, 4, 6, 8};
    int max_threads = 0;
    // with the library's choice of kernel, the interpreter competes with the
    // tape-specialised kernel; candidates are generated (and timed) with the
    // problem switched to the kernel they use
    std::vector<bool> kernels{false};
    if (use_jit(p) && p->opt.specialize == -1) kernels.push_back(true);
    for (bool ip : kernels) {
    p->tuned_interp = ip;
    for (bool sy : sync_choices(p))
    for (int t : tpsub_choices(p))
        for (int b : blocks)
            for (int k : bpss) {
                const int warps = b * k / 32;
                if (warps < 4 || warps > 32 || !groups_fit(b, t)) continue;
                if (b > (reduce_jit(p) ? p->jit.block_max : kInterpBlockMax)) continue;
                for (int sm = 0; sm < 2; ++sm) {
                    const size_t bytes = smem_bytes(p, b, sm);
                    if (sm && (reduce_jit(p) || bytes + 1024 > (size_t)p->smem_optin || bytes * k > 220 * 1024)) continue;
                    if (p->opt.frame_in_shared == 0 && sm) continue;
                    if (p->opt.frame_in_shared == 1 && !sm && !reduce_jit(p)) continue;
                    if (reduce_occupancy(p, b, sm, t, sy) < k) continue;
                    cands.push_back({b, k, sm, t, 1, sy, ip});
                    max_threads = std::max(max_threads, b * k * p->sm_count);
                }
            }
    }
    p->tuned_interp = false;
    if (cands.empty()) cands.push_back({64, 1, 0, 1, 1, false, false});
    // time only [0, cap) of the global index range: two waves of the widest candidate grid
    const long long cap = std::min<long long>(total, std::max<long long>(2LL * max_threads, 1LL << 18));
    long long* hdr = reinterpret_cast<long long*>(p->h_queue);
    const long long g_end = hdr[1];
    CK(cudaEventSynchronize(p->queue_free));
    hdr[1] = cap;
    CK(cudaMemcpyAsync(p->d_queue, p->h_queue, 16, cudaMemcpyHostToDevice, s));
    cudaEvent_t ew, e0, e1;
    CK(cudaEventCreate(&ew));
    CK(cudaEventCreate(&e0));
    CK(cudaEventCreate(&e1));
    float best = 1e30f, worst = 0.f, last_ms = 0.f;
    TuneCand bc = cands[0];
    ivb_status st = IVB_OK;
    int timed = 0;
    auto time_one = [&](const TuneCand& c) -> ivb_status {
        const int grid = p->sm_count * c.bps;
        p->tuned_interp = c.interp;
        ivb_status r = IVB_OK;
        if (reduce_units(p) > 0) r = ensure_frame(p, grid, c.block, reduce_units(p));
        if (r == IVB_ENOMEM) { p->err.clear(); last_ms = 1e30f; return IVB_OK; }   // not a choice: left out
        if (r) return r;
        const int tile = c.tile_mult * pass_size(p, c.block, c.tpsub);
        // warm-up run, timed too: a candidate whose warm-up already takes 1.5x the
        // best time so far is not run again (its warm-up time stands)
        CK(cudaEventRecord(ew, s));
        r = enqueue_bound(p, grid, c.block, tile, c.smem, p->max_nodes, s, c.tpsub, c.sync);
        if (r) return r;
        CK(cudaEventRecord(e0, s));
        CK(cudaEventSynchronize(e0));
        float ms = 0;
        CK(cudaEventElapsedTime(&ms, ew, e0));
        if (!(best < 1e29f && ms > 1.5f * best)) {
            r = enqueue_bound(p, grid, c.block, tile, c.smem, p->max_nodes, s, c.tpsub, c.sync);
            if (r) return r;
            CK(cudaEventRecord(e1, s));
            CK(cudaEventSynchronize(e1));
            CK(cudaEventElapsedTime(&ms, e0, e1));
        }
        ++timed;
        last_ms = ms;
        worst = std::max(worst, ms);
        if (ms < best) { best = ms; bc = c; }
        return IVB_OK;
    };
    // Blocks come largest first. When the best launch of one block size takes over
    // twice the best time so far, smaller blocks of the same kernel are left out:
    // their warps share even less code (configuration 5: 68 launches in 16 s, now 47 in
    // 4 s).
    float size_ms = 1e30f;      // best time of the block size being timed
    bool hopeless = false;
    for (size_t i = 0; i < cands.size() && !st; ++i) {
        const TuneCand& c = cands[i];
        const bool same = i > 0 && cands[i - 1].interp == c.interp && cands[i - 1].sync == c.sync && cands[i - 1].tpsub == c.tpsub;
        if (!same) hopeless = false;
        else if (cands[i - 1].block != c.block) hopeless = hopeless || (size_ms < 1e29f && size_ms > 2.f * best);
        if (!same || cands[i - 1].block != c.block) size_ms = 1e30f;
        if (hopeless) continue;
        st = time_one(c);
        size_ms = std::min(size_ms, last_ms);
    }
    // larger grabs: not for segmented kernels, whose passes are long and dealt out
    // evenly (a grab of four passes that fits the sample leaves others unbalanced)
    if (!st && timed > 0 && p->opt.tile <= 0 && (bc.interp || p->jit.state_units == 0)) {
        const TuneCand base = bc;
        for (int mult : {4, 16}) {
            TuneCand c = base;
            c.tile_mult = mult;
            st = time_one(c);
            if (st) break;
        }
    }
    p->tuned_interp = false;
    cudaEventDestroy(ew);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    // restore the batch's index range
    hdr[1] = g_end;
    CK(cudaMemcpyAsync(p->d_queue, p->h_queue, 16, cudaMemcpyHostToDevice, s));
    CK(cudaStreamSynchronize(s));
    if (!st && timed == 0) {   // no candidate's frames fit: the default shape, on as many blocks as do
        st = default_tuning(p);
        p->tuned = true;
    }
    if (st || timed == 0) return st;
    p->block = bc.block;
    p->bps = bc.bps;
    p->frame_smem = bc.smem;
    p->tpsub = bc.tpsub;
    p->chunk_sync = bc.sync;
    p->tuned_interp = bc.interp;
    p->tile = bc.tile_mult * pass_size(p, bc.block, bc.tpsub);
    p->tune_candidates = timed;
    p->tune_best_ms = best;
    p->tune_worst_ms = worst;
    p->tuned = true;
    p->cfg_ready = true;
    drop_graphs(p);
    // the widest candidate's frames go back where the choice needs less
    if ((size_t)p->sm_count * p->block * p->bps * reduce_units(p) * sizeof(double) < p->frame_bytes) free_frame(p);
    return IVB_OK;
}

bool wide(const ivb_problem* p, int units) { return wide_frames_fit(units * sizeof(double), p->sm_count, p->device_bytes); }

ivb_status default_tuning(ivb_problem* p) {
    // a segmented kernel runs best as one block per SM: its warps then stream
    // through the same code (configuration 5, 2^19 subdomains: 1024-thread
    // blocks 56 ms, 2 x 512 71 ms, 4 x 256 118 ms)
    const bool seg = reduce_jit(p) && p->jit.state_units > 0;
    // the interpreter: frames in shared memory if four small blocks' fit, else 32
    // warps per SM (configuration 3, 941192 subdomains: 12.8 ms against 17.2 with 16)
    const bool small = reduce_jit(p) || p->opt.frame_in_shared != -1 || !wide(p, frame_units(p)) ||
                       (smem_bytes(p, 128, 1) + 1024 <= (size_t)p->smem_optin && smem_bytes(p, 128, 1) * 4 <= 220 * 1024);
    const int seg_block = wide(p, p->jit.state_units) ? p->jit.block_max : std::min(512, p->jit.block_max);
    p->block = p->opt.block_threads > 0 ? p->opt.block_threads : seg ? seg_block : small ? 128 : 256;
    if (!reduce_jit(p)) p->block = std::min(p->block, kInterpBlockMax);   // asked of a kernel that did not compile
    p->bps = p->opt.blocks_per_sm > 0 ? p->opt.blocks_per_sm : seg && p->opt.block_threads <= 0 ? 1 : 4;
    const size_t bytes = smem_bytes(p, p->block, 1);
    if (reduce_jit(p)) p->frame_smem = 0;   // frames serve only the interpreter's store mode
    else if (p->opt.frame_in_shared == 1) p->frame_smem = 1;
    else if (p->opt.frame_in_shared == 0) p->frame_smem = 0;
    else p->frame_smem = (bytes + 1024 <= (size_t)p->smem_optin && bytes * p->bps <= 220 * 1024) ? 1 : 0;
    p->tpsub = block_tpsub(p->block, tpsub_choices(p).front());
    p->chunk_sync = sync_choices(p).front();
    const int occ = reduce_occupancy(p, p->block, p->frame_smem, p->tpsub, p->chunk_sync);
    if (occ < 1) return fail(p, IVB_ENOTSUP, "launch configuration does not fit on an SM");
    if (p->bps > occ) p->bps = occ;
    const int per = pass_size(p, p->block, p->tpsub);
    p->tile = p->opt.tile > 0 ? ((p->opt.tile + per - 1) / per) * per : per;
    p->cfg_ready = true;
    const bool explicit_cfg = p->opt.block_threads > 0 || p->opt.blocks_per_sm > 0;
    if (!p->opt.autotune || explicit_cfg) p->tuned = true;
    return IVB_OK;
}

// Where a call's node results go. k_finalize writes straight to device arrays of
// this device; what the host wants is packed in d_out and comes over in one copy.
// Anything else (another device, managed memory, an unaligned address) is copied
// array by array.
struct Outputs {
    struct Item { void* user; size_t offset, bytes; bool direct, host; } it[5];
    OutLayout L;
    bool any_host = false;

    Outputs(ivb_problem* p, int n_nodes, double* lb, uint8_t* inf, double* ub, double* minlo, double* maxhi,
            QueueHeader* H, char* d_out)
        : L(n_nodes, minlo || maxhi ? p->n_out : 0) {
        const size_t n = n_nodes, hull = n * p->n_out * sizeof(double);
        it[0] = {lb, 0, n * sizeof(double), false, false};
        it[1] = {ub, L.ub, n * sizeof(double), false, false};
        it[2] = {minlo, L.minlo, hull, false, false};
        it[3] = {maxhi, L.maxhi, hull, false, false};
        it[4] = {inf, L.inf, n, false, false};
        void* at[5];
        for (int k = 0; k < 5; ++k) {
            Item& x = it[k];
            at[k] = nullptr;
            if (!x.user) continue;
            cudaPointerAttributes a;
            const bool ok = cudaPointerGetAttributes(&a, x.user) == cudaSuccess;
            if (!ok) cudaGetLastError();
            const bool dev = ok && (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged);
            x.direct = dev && a.type == cudaMemoryTypeDevice && a.device == p->device &&
                       (k == 4 || reinterpret_cast<uintptr_t>(x.user) % sizeof(double) == 0);
            x.host = !dev;
            any_host |= x.host;
            at[k] = x.direct ? x.user : d_out + x.offset;
        }
        H->lb = static_cast<double*>(at[0]);
        H->ub = static_cast<double*>(at[1]);
        H->minlo = static_cast<double*>(at[2]);
        H->maxhi = static_cast<double*>(at[3]);
        H->inf = static_cast<uint8_t*>(at[4]);
    }

    // after the kernels are enqueued: copies, and the wait that host arrays need
    ivb_status deliver(ivb_problem* p, const char* d_out, cudaStream_t s) const {
        const bool packed = any_host && L.bytes <= kPinnedMost;
        if (packed) {
            const ivb_status st = ensure_pinned(p, p->h_out, L.bytes);
            if (st) return st;
            CK(cudaMemcpyAsync(p->h_out.p, d_out, L.bytes, cudaMemcpyDeviceToHost, s));
        }
        for (const Item& x : it) {
            if (!x.user || x.direct || (x.host && packed)) continue;
            CK(cudaMemcpyAsync(x.user, d_out + x.offset, x.bytes, x.host ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice, s));
        }
        if (!any_host) return IVB_OK;
        CK(cudaStreamSynchronize(s));
        if (packed)
            for (const Item& x : it)
                if (x.user && x.host) std::memcpy(x.user, p->h_out.p + x.offset, x.bytes);
        return IVB_OK;
    }
};

}  // namespace

// ======================================================================= ABI

// interval operations per subdomain
long long interval_ops(const HostProgram& P, int grad_mode) {
    const int64_t* cnt = grad_mode == IVB_GRAD_ADJOINT ? P.cnt_adj : P.cnt_fwd;
    long long ends = 0;
    for (int k = 0; k < IVB_CNT_N; ++k) ends += cnt[k];
    return ends / 2;
}

// segmentation options of a problem
SegPolicy seg_policy(const ivb_options& o, const HostProgram& P) {
    SegPolicy pol;
    if (o.recompute >= 0) pol.recompute = o.recompute;
    if (o.seg_chunk > 0) pol.chunk_cost = o.seg_chunk;
    if (o.seg_ilp > 0) pol.ilp = o.seg_ilp;
    const int emu = o.emulate >= 0 ? o.emulate : kJitDefaultEmulate;
    pol.outline = seg_outline_for(o.seg_outline, emu, interval_ops(P, IVB_GRAD_ADJOINT));
    pol.max_regs = seg_budget(o.seg_regs, o.block_threads, o.blocks_per_sm);
    const unsigned hc = std::thread::hardware_concurrency();
    pol.units = std::max(1, std::min(64, hc ? (int)hc : 8));
    return pol;
}

cudaError_t specialize_seg(ivb_problem* p, const std::vector<Ins>& ins, const std::vector<RIns>& rins,
                           const std::vector<double>& consts, std::string* msg) {
    const int emu = p->opt.emulate >= 0 ? p->opt.emulate : kJitDefaultEmulate;
    const SegPolicy pol = seg_policy(p->opt, p->P);
    const int block_max = seg_block_max(pol.max_regs);
    const SegSource src = jit_seg_source(p->P, ins, rins, consts, block_max, emu, p->opt.form, pol);
    std::vector<char> cubin;
    std::string tables;
    double secs = 0.0;
    *msg = jit_seg_compile(src, pol.max_regs, cubin, tables, &secs, nullptr, nullptr);
    if (!msg->empty()) return cudaSuccess;
    cudaError_t ce = jit_load(cubin, tables, p->jit);
    if (ce != cudaSuccess) return ce;
    p->jit.kern_t[0] = p->jit.kern;
    for (int t : src.ts) {
        const std::string name = "ivb_jit_bound_t" + std::to_string(t);
        if (t > 1) {
            ce = cudaLibraryGetKernel(&p->jit.kern_t[tpsub_index(t)], p->jit.lib, name.c_str());
            if (ce != cudaSuccess) return ce;
        }
        ce = cudaLibraryGetKernel(&p->jit.kern_sync[tpsub_index(t)], p->jit.lib, (name + "_sync").c_str());
        if (ce != cudaSuccess) return ce;
    }
    p->jit.mode = KM_ADJ_REDUCE;
    p->jit.emulate = emu;
    p->jit.compact = true;
    p->jit.block_max = block_max;
    p->jit.compile_seconds = secs;
    p->jit.state_units = src.state_units;
    p->jit.chunks = src.chunks;
    p->jit.state_loads = src.loads;
    p->jit.state_stores = src.stores;
    p->jit.recomputed = src.recomputed;
    p->jit.recompute = pol.recompute;
    p->jit.ilp = src.ilp;
    return cudaSuccess;
}

// generate, compile and load the tape-specialised reduce kernel
cudaError_t specialize(ivb_problem* p, const std::vector<Ins>& ins, const std::vector<RIns>& rins,
                       const std::vector<double>& consts, int mode, std::string* msg) {
    const int emu = p->opt.emulate >= 0 ? p->opt.emulate : kJitDefaultEmulate;
    const bool compact = p->opt.specialize != 2;
    const std::string src =
        jit_source(p->P, ins, rins, consts, mode, kJitBlockMax, kJitMinBlocks, emu, compact, p->opt.form);
    std::vector<char> cubin;
    std::string tables;
    double secs = 0.0;
    *msg = jit_compile(src, cubin, tables, &secs, nullptr, nullptr);
    if (!msg->empty()) return cudaSuccess;
    const cudaError_t ce = jit_load(cubin, tables, p->jit);
    if (ce != cudaSuccess) return ce;
    p->jit.mode = mode;
    p->jit.emulate = emu;
    p->jit.compact = compact;
    p->jit.block_max = kJitBlockMax;
    p->jit.compile_seconds = secs;
    return cudaSuccess;
}

extern "C" void ivb_options_default(ivb_options* o) {
    if (!o) return;
    o->grad_mode = IVB_GRAD_ADJOINT;
    o->form = IVB_FORM_MVF;
    o->filter = 0;
    o->batched = 1;
    o->use_graph = 1;
    o->autotune = 1;
    o->block_threads = 0;
    o->blocks_per_sm = 0;
    o->tile = 0;
    o->max_nodes = 4096;
    o->frame_in_shared = -1;
    o->specialize = 0;
    o->emulate = -1;
    o->recompute = -1;
    o->seg_chunk = 0;
    o->seg_regs = 0;
    o->threads_per_subdomain = 0;
    o->seg_sync = -1;
    o->seg_ilp = 0;
    o->seg_outline = -1;
}

extern "C" ivb_status ivb_create_problem(const ivb_tape* tape, const ivb_options* opt, ivb_problem** out) {
    if (!out) return fail(nullptr, IVB_EINVAL, "out is NULL");
    *out = nullptr;
    std::string e = validate_tape(tape);
    if (!e.empty()) return fail(nullptr, IVB_ETAPE, e);
    ivb_options o;
    ivb_options_default(&o);
    if (opt) o = *opt;
    if (o.grad_mode != IVB_GRAD_FORWARD && o.grad_mode != IVB_GRAD_ADJOINT)
        return fail(nullptr, IVB_EINVAL, "grad_mode must be IVB_GRAD_FORWARD or IVB_GRAD_ADJOINT");
    if (o.form < 0 || o.form > 2) return fail(nullptr, IVB_EINVAL, "form must be 0, 1 or 2");
    if (o.max_nodes < 1 || o.max_nodes > (1 << 20)) return fail(nullptr, IVB_EINVAL, "max_nodes must be in [1, 2^20]");
    if (o.block_threads < 0 || (o.block_threads % 32))
        return fail(nullptr, IVB_EINVAL, "block_threads must be a multiple of 32 (0 = auto)");
    if (o.specialize < -1 || o.specialize > 3) return fail(nullptr, IVB_EINVAL, "specialize must be -1, 0, 1, 2 or 3");
    if (o.specialize == 3 && o.grad_mode != IVB_GRAD_ADJOINT)
        return fail(nullptr, IVB_EINVAL, "specialize = 3 (segmented) needs grad_mode IVB_GRAD_ADJOINT");
    if (o.recompute < -1 || o.recompute > 2) return fail(nullptr, IVB_EINVAL, "recompute must be -1, 0, 1 or 2");
    if (o.seg_chunk < 0 || o.seg_chunk > 100000) return fail(nullptr, IVB_EINVAL, "seg_chunk must be in [0, 100000]");
    if (o.threads_per_subdomain != 0 && o.threads_per_subdomain != 1 && o.threads_per_subdomain != 2 &&
        o.threads_per_subdomain != 4)
        return fail(nullptr, IVB_EINVAL, "threads_per_subdomain must be 0 (tuned), 1, 2 or 4");
    if (o.seg_sync < -1 || o.seg_sync > 1) return fail(nullptr, IVB_EINVAL, "seg_sync must be -1, 0 or 1");
    if (o.seg_ilp < 0 || o.seg_ilp > 2) return fail(nullptr, IVB_EINVAL, "seg_ilp must be 0, 1 or 2");
    if (o.seg_outline < -1 || o.seg_outline > 2) return fail(nullptr, IVB_EINVAL, "seg_outline must be -1, 0, 1 or 2");
    if (o.seg_regs != 0 && (o.seg_regs < 64 || o.seg_regs > 255))
        return fail(nullptr, IVB_EINVAL, "seg_regs must be 0 or in [64, 255]");
    if (o.emulate < -1 || o.emulate > 15) return fail(nullptr, IVB_EINVAL, "emulate must be -1 or a bitmask in [0, 15]");
    ivb_problem* p = new ivb_problem();
    p->opt = o;
    std::vector<Ins> ins;
    std::vector<RIns> rins;
    std::vector<double> consts;
    e = compile_tape(tape, p->P, ins, rins, consts);
    if (!e.empty()) { delete p; return fail(nullptr, IVB_ENOTSUP, e); }
    // the kernel, and the largest block that options can ask of it: every shape that the
    // autotuner reports can be asked for
    const bool small = interval_ops(p->P, o.grad_mode) <= (o.grad_mode == IVB_GRAD_ADJOINT ? kSegMinOps : kJitAutoMaxOps);
    const bool seg = o.specialize == 3 || (o.specialize == -1 && !small && o.grad_mode == IVB_GRAD_ADJOINT);
    const int most = seg ? seg_block_limit(o.seg_regs) : o.specialize >= 1 ? kCompiledBlockMax : kInterpBlockMax;
    if (o.block_threads > most) {
        delete p;
        return fail(nullptr, IVB_EINVAL, "block_threads above " + std::to_string(most) + " with this kernel");
    }
    // by the library's choice, a block beyond the compiled kernel's runs the interpreter
    const bool compiled = seg || o.specialize >= 1 || (o.specialize == -1 && small && o.block_threads <= kCompiledBlockMax);
    p->n = tape->n_vars;
    p->n_out = tape->n_outputs;
    p->obj = p->P.obj;
    for (int i = 0; i < p->n_out; ++i) p->out_kind[i] = tape->out_kind[i];
    p->max_nodes = o.max_nodes;
    p->rec_bytes = queue_rec_bytes(p->n);
    host_tape(tape, p->host);

    auto bail = [&](cudaError_t ce, const char* where) {
        std::string m = std::string(where) + ": " + cudaGetErrorString(ce);
        ivb_destroy(p);
        return fail(nullptr, ce == cudaErrorMemoryAllocation ? IVB_ENOMEM : IVB_ECUDA, m);
    };
#define CKC(call)                                   \
    do {                                            \
        cudaError_t e_ = (call);                    \
        if (e_ != cudaSuccess) return bail(e_, #call); \
    } while (0)
    int dev = 0;
    CKC(cudaGetDevice(&dev));
    p->device = dev;
    CKC(cudaDeviceGetAttribute(&p->sm_count, cudaDevAttrMultiProcessorCount, dev));
    CKC(cudaDeviceGetAttribute(&p->smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    size_t unused = 0;
    CKC(cudaMemGetInfo(&unused, &p->device_bytes));
    for (int m = 0; m < 4; ++m) CKC(set_bound_smem_limit(m, p->smem_optin - 1024));
    CKC(init_math_tables());

    CKC(cudaMalloc(&p->d_consts, std::max<size_t>(1, consts.size()) * sizeof(double)));
    if (!consts.empty())
        CKC(cudaMemcpy(p->d_consts, consts.data(), consts.size() * sizeof(double), cudaMemcpyHostToDevice));
    std::vector<XIns> xins, pins;
    std::vector<XRIns> xrins, prins;
    interpreter_programs(p->P, ins, rins, xins, xrins);
    CKC(cudaMalloc(&p->d_xins, xins.size() * sizeof(XIns)));
    CKC(cudaMalloc(&p->d_xrins, xrins.size() * sizeof(XRIns)));
    CKC(cudaMemcpy(p->d_xins, xins.data(), xins.size() * sizeof(XIns), cudaMemcpyHostToDevice));
    CKC(cudaMemcpy(p->d_xrins, xrins.data(), xrins.size() * sizeof(XRIns), cudaMemcpyHostToDevice));
    const size_t xtan = ins.size();
    p->point_units = point_programs(p->P, ins, rins, pins, prins);
    CKC(cudaMalloc(&p->d_pins, pins.size() * sizeof(XIns)));
    CKC(cudaMalloc(&p->d_prins, prins.size() * sizeof(XRIns)));
    CKC(cudaMemcpy(p->d_pins, pins.data(), pins.size() * sizeof(XIns), cudaMemcpyHostToDevice));
    CKC(cudaMemcpy(p->d_prins, prins.data(), prins.size() * sizeof(XRIns), cudaMemcpyHostToDevice));
    ProgDesc D{};
    std::vector<uint32_t> masks;
    tangent_masks(p->P, ins, masks, D.tan_out_mask);
    CKC(cudaMalloc(&p->d_tan_mask, masks.size() * sizeof(uint32_t)));
    CKC(cudaMemcpy(p->d_tan_mask, masks.data(), masks.size() * sizeof(uint32_t), cudaMemcpyHostToDevice));
    D.tan_mask = reinterpret_cast<const uint2*>(p->d_tan_mask);
    D.pins = p->d_pins;
    D.prins = p->d_prins;
    D.xins = p->d_xins;
    D.xtan = p->d_xins + xtan;
    D.xcone = D.xtan + p->P.tan_count;
    D.xrins = p->d_xrins;
    D.consts = p->d_consts;
    D.n = p->n;
    D.n_out = p->n_out;
    D.obj = p->obj;
    D.has_eq = p->P.has_eq;
    D.pt_begin = p->P.pt_begin;
    D.pt_count = p->P.pt_count;
    D.tan_begin = p->P.tan_begin;
    D.tan_count = p->P.tan_count;
    for (int i = 0; i < p->n_out; ++i) {
        D.pt_out_ref[i] = (uint32_t)p->P.pt_out_ref[i];
        D.pt_out_kind[i] = (uint32_t)p->P.pt_out_kind[i];
        D.tan_out_ref[i] = (uint32_t)p->P.tan_out_ref[i];
        D.tan_out_kind[i] = (uint32_t)p->P.tan_out_kind[i];
        D.adj[i] = p->P.adj[i];
        D.out_kind[i] = p->out_kind[i];
    }
    D.L = p->P.L;
    CKC(cudaMalloc(&p->d_prog, sizeof(ProgDesc)));
    CKC(cudaMemcpy(p->d_prog, &D, sizeof(ProgDesc), cudaMemcpyHostToDevice));
    CKC(cudaMalloc(&p->d_out_kind, 64));
    CKC(cudaMemcpy(p->d_out_kind, p->out_kind, 64, cudaMemcpyHostToDevice));

    const size_t qb = queue_bytes(p->max_nodes, p->n);
    CKC(cudaMalloc(&p->d_queue, qb));
    CKC(cudaMallocHost(&p->h_queue, qb));
    CKC(cudaEventCreateWithFlags(&p->queue_free, cudaEventDisableTiming));
    CKC(cudaEventRecord(p->queue_free, 0));
    CKC(cudaMalloc(&p->d_keys, (size_t)p->max_nodes * (2 * p->n_out + 2) * sizeof(unsigned long long)));
    CKC(cudaMalloc(&p->d_counter, sizeof(unsigned long long)));
    CKC(cudaMalloc(&p->d_out, OutLayout(p->max_nodes, p->n_out).bytes));
    CKC(cudaStreamCreateWithFlags(&p->cap_stream, cudaStreamNonBlocking));
    if (compiled) {
        const int mode = o.grad_mode == IVB_GRAD_ADJOINT ? KM_ADJ_REDUCE : KM_FWD_REDUCE;
        std::string msg;
        const cudaError_t ce = seg ? specialize_seg(p, ins, rins, consts, &msg)
                                   : specialize(p, ins, rins, consts, mode, &msg);
        if (ce != cudaSuccess || !msg.empty()) {
            jit_unload(p->jit);
            if (o.specialize >= 1) {
                ivb_destroy(p);
                if (ce != cudaSuccess)
                    return fail(nullptr, ce == cudaErrorMemoryAllocation ? IVB_ENOMEM : IVB_ECUDA,
                                std::string("loading the tape-specialised kernel: ") + cudaGetErrorString(ce));
                return fail(nullptr, IVB_ENOTSUP, msg);
            }
            cudaGetLastError();
        }
    }
#undef CKC
    *out = p;
    return IVB_OK;
}

ivb_status ensure_pinned(ivb_problem* p, ivb_problem::Pinned& P, size_t bytes) {
    if (bytes <= P.bytes) return IVB_OK;
    if (P.p) cudaFreeHost(P.p);
    P.p = nullptr;
    P.bytes = 0;
    const size_t want = std::max<size_t>(2 * bytes, 4096);
    CK(cudaMallocHost(&P.p, want));
    P.bytes = want;
    return IVB_OK;
}

namespace {
ivb_status bound_nodes_impl(ivb_problem* p, int32_t n_nodes, const double* boxes, const int32_t* splits_per_dim,
                            double* out_lb, uint8_t* out_infeasible, double* out_ub, double* out_minlo,
                            double* out_maxhi, char* packed, cudaStream_t s);
}  // namespace

extern "C" ivb_status ivb_bound_nodes_ex(ivb_problem* p, int32_t n_nodes, const double* boxes,
                                         const int32_t* splits_per_dim, double* out_lb, uint8_t* out_infeasible,
                                         double* out_ub, double* out_minlo, double* out_maxhi, void* cuda_stream) {
    return bound_nodes_impl(p, n_nodes, boxes, splits_per_dim, out_lb, out_infeasible, out_ub, out_minlo, out_maxhi,
                            nullptr, (cudaStream_t)cuda_stream);
}

ivb_status bound_nodes_enqueue(ivb_problem* p, int32_t n_nodes, const double* boxes, const int32_t* splits,
                               char* packed, cudaStream_t s) {
    return bound_nodes_impl(p, n_nodes, boxes, splits, nullptr, nullptr, nullptr, nullptr, nullptr, packed, s);
}

namespace {
// packed: results of the nodes go there in one copy, without a wait (bound_nodes_enqueue)
ivb_status bound_nodes_impl(ivb_problem* p, int32_t n_nodes, const double* boxes, const int32_t* splits_per_dim,
                            double* out_lb, uint8_t* out_infeasible, double* out_ub, double* out_minlo,
                            double* out_maxhi, char* packed, cudaStream_t s) {
    if (!p) return fail(nullptr, IVB_EINVAL, "problem handle is NULL");
    p->err.clear();
    if (n_nodes == 0) return IVB_OK;   // empty batch: nothing to bound
    if (n_nodes < 0 || n_nodes > p->max_nodes)
        return fail(p, IVB_EINVAL, "n_nodes must be in [0, max_nodes]");
    if (!boxes || !splits_per_dim) return fail(p, IVB_EINVAL, "boxes and splits_per_dim must not be NULL");
    size_t qbytes = 0;
    long long total = 0;
    ivb_status st = stage_queue(p, n_nodes, boxes, splits_per_dim, 0, 0, false, &qbytes, &total, s);
    if (st) return st;
    QueueHeader* H = reinterpret_cast<QueueHeader*>(p->h_queue);
    const Outputs out(p, n_nodes, out_lb, out_infeasible, out_ub, out_minlo, out_maxhi, H, p->d_out);
    if (packed) {
        const OutLayout L(n_nodes, 0);
        H->lb = reinterpret_cast<double*>(p->d_out);
        H->ub = reinterpret_cast<double*>(p->d_out + L.ub);
        H->inf = reinterpret_cast<uint8_t*>(p->d_out + L.inf);
    }

    if (!p->opt.batched) {
        // plain path: one node per launch, node queue of one record each
        if (!p->cfg_ready) { st = default_tuning(p); if (st) return st; }
        const int n = p->n;
        std::vector<char> one(queue_bytes(1, n));
        const char* q = p->h_queue;
        const long long* off = reinterpret_cast<const long long*>(q + kQueueHeader);
        const char* recs = q + kQueueHeader + 8 * (size_t)(n_nodes + 1);
        for (int nd = 0; nd < n_nodes; ++nd) {
            // build a one-node queue in place at the front of the device buffer
            long long hdr[2] = {1, off[nd + 1] - off[nd]};
            long long o2[2] = {0, off[nd + 1] - off[nd]};
            std::memset(one.data(), 0, kQueueHeader);
            std::memcpy(one.data(), hdr, sizeof(hdr));
            std::memcpy(one.data() + kQueueHeader, o2, sizeof(o2));
            std::memcpy(one.data() + kQueueHeader + 16, recs + (size_t)nd * p->rec_bytes, p->rec_bytes);
            CK(cudaMemcpyAsync(p->d_queue, one.data(), one.size(), cudaMemcpyHostToDevice, s));
            const long long S = o2[1];
            const long long tiles = (S + p->block - 1) / p->block;
            int grid = (int)std::min<long long>(tiles, (long long)p->sm_count * p->bps);
            st = fit_frame(p, &grid, p->block, reduce_units(p));
            if (st) return st;
            CK(launch_init_keys(p->d_keys, p->d_queue, 1, p->n_out, p->d_counter, s));
            KParams K = make_params(p, p->frame_smem);
            K.tile = pass_size(p, p->block, p->tpsub);
            CK(launch_reduce(p, K, grid, p->block, p->frame_smem, s, p->tpsub, p->chunk_sync));
            FinalizeParams F{};
            F.keys = p->d_keys; F.queue = p->d_queue; F.max_nodes = 1; F.n_out = p->n_out; F.obj = p->obj;
            F.filter = p->opt.filter; F.out_kind = p->d_out_kind;
            if (H->lb) F.lb = H->lb + nd;
            if (H->inf) F.inf = H->inf + nd;
            if (H->ub) F.ub = H->ub + nd;
            if (H->minlo) F.minlo = H->minlo + (size_t)nd * p->n_out;
            if (H->maxhi) F.maxhi = H->maxhi + (size_t)nd * p->n_out;
            CK(launch_finalize(F, s));
            p->launches += 3;
            // the host buffer `one` is reused: wait for this node's copy
            CK(cudaStreamSynchronize(s));
        }
        CK(cudaEventRecord(p->queue_free, s));
    } else {
        CK(cudaMemcpyAsync(p->d_queue, p->h_queue, qbytes, cudaMemcpyHostToDevice, s));
        CK(cudaEventRecord(p->queue_free, s));
        if (!p->tuned) {
            // tune on the first batch with enough work to time; defaults until then
            const bool explicit_cfg = p->opt.block_threads > 0 || p->opt.blocks_per_sm > 0;
            if (p->opt.autotune && !explicit_cfg && total >= (1LL << 18)) st = autotune(p, total, s);
            else if (!p->cfg_ready) st = default_tuning(p);
            if (st) return st;
        }
        int grid = p->sm_count * p->bps;
        st = fit_frame(p, &grid, p->block, reduce_units(p));
        if (st) return st;
        const int tpsub = call_tpsub(p, total, (long long)grid * p->block);
        const int tile = tpsub == p->tpsub ? p->tile : pass_size(p, p->block, tpsub);
        if (p->opt.use_graph) {
            cudaGraphExec_t& gexec = p->gexec[tpsub_index(tpsub)];
            if (!gexec) {
                cudaGraph_t g = nullptr;
                CK(cudaStreamBeginCapture(p->cap_stream, cudaStreamCaptureModeThreadLocal));
                st = enqueue_bound(p, grid, p->block, tile, p->frame_smem, p->max_nodes, p->cap_stream, tpsub,
                                   p->chunk_sync);
                cudaGraph_t gg = nullptr;
                cudaError_t ce = cudaStreamEndCapture(p->cap_stream, &gg);
                if (st) { if (gg) cudaGraphDestroy(gg); return st; }
                if (ce != cudaSuccess) return cuda_fail(p, ce, "cudaStreamEndCapture");
                g = gg;
                ce = cudaGraphInstantiate(&gexec, g, 0);
                cudaGraphDestroy(g);
                if (ce != cudaSuccess) { gexec = nullptr; return cuda_fail(p, ce, "cudaGraphInstantiate"); }
                p->launches -= 3;   // captured, not launched
            }
            CK(cudaGraphLaunch(gexec, s));
            p->launches += 3;
        } else {
            st = enqueue_bound(p, grid, p->block, tile, p->frame_smem, p->max_nodes, s, tpsub, p->chunk_sync);
            if (st) return st;
        }
    }
    if (packed) {
        CK(cudaMemcpyAsync(packed, p->d_out, OutLayout(n_nodes, 0).bytes, cudaMemcpyDeviceToHost, s));
        return IVB_OK;
    }
    return out.deliver(p, p->d_out, s);
}
}  // namespace

extern "C" ivb_status ivb_bound_nodes(ivb_problem* p, int32_t n_nodes, const double* boxes,
                                      const int32_t* splits_per_dim, double* out_lb, uint8_t* out_infeasible,
                                      void* cuda_stream) {
    return ivb_bound_nodes_ex(p, n_nodes, boxes, splits_per_dim, out_lb, out_infeasible, nullptr, nullptr, nullptr,
                              cuda_stream);
}

extern "C" ivb_status ivb_enclose(ivb_problem* p, const double* box, const int32_t* splits_per_dim, int64_t first,
                                  int64_t count, double* out_F, double* out_Fc, double* out_G, void* cuda_stream) {
    if (!p) return fail(nullptr, IVB_EINVAL, "problem handle is NULL");
    p->err.clear();
    if (!box || !splits_per_dim || !out_F) return fail(p, IVB_EINVAL, "box, splits and out_F must not be NULL");
    if (count < 1 || count > (1LL << 24)) return fail(p, IVB_EINVAL, "count must be in [1, 2^24]");
    cudaStream_t s = (cudaStream_t)cuda_stream;
    size_t qbytes = 0;
    long long total = 0;
    ivb_status st = stage_queue(p, 1, box, splits_per_dim, first, count, true, &qbytes, &total, s);
    if (st) return st;
    if (!p->cfg_ready) { st = default_tuning(p); if (st) return st; }
    CK(cudaMemcpyAsync(p->d_queue, p->h_queue, qbytes, cudaMemcpyHostToDevice, s));
    CK(cudaEventRecord(p->queue_free, s));
    const int n_out = p->n_out, n = p->n;
    const size_t fb = (size_t)count * n_out * 2 * sizeof(double), gb = fb * n;
    // outputs: written directly when device pointers, else through device temporaries
    const bool dF = is_device_ptr(out_F), dFc = out_Fc && is_device_ptr(out_Fc), dG = out_G && is_device_ptr(out_G);
    double *tF = nullptr, *tFc = nullptr, *tG = nullptr;
    if (!dF) CK(cudaMallocAsync(&tF, fb, s));
    if (out_Fc && !dFc) CK(cudaMallocAsync(&tFc, fb, s));
    if (out_G && !dG) CK(cudaMallocAsync(&tG, gb, s));
    const unsigned long long first_u = (unsigned long long)first;
    CK(cudaMemcpyAsync(p->d_counter, &first_u, sizeof(first_u), cudaMemcpyHostToDevice, s));
    // the store modes run the interpreter: in the shape of the reduce launches where these run it too,
    // else in the options' or its own
    const bool own = !reduce_jit(p);
    const int asked = std::min(p->opt.block_threads, kInterpBlockMax);
    const int block = own ? p->block : asked > 0 ? asked : wide(p, frame_units(p)) ? 256 : 128;
    const int bps = own ? p->bps : p->opt.blocks_per_sm > 0 ? p->opt.blocks_per_sm : 4;
    const int fs = own ? p->frame_smem : 0;
    const int resident = p->sm_count * bps;
    int grid = range_blocks(count, resident);   // dealt out evenly
    st = fit_frame(p, &grid, block, frame_units(p));
    if (st) return st;
    KParams K = make_params(p, fs);
    K.frame_units = frame_units(p);
    // few subdomains: the outputs of each are shared among 2, 4 or 8 warp groups, as
    // long as all warps are resident (the warps run latency-bound; 50003
    // subdomains of configuration 3, 6 outputs: 1.38 -> 1.03 ms)
    K.groups = 1;
    if (p->opt.grad_mode == IVB_GRAD_ADJOINT)
        while (2 * K.groups <= std::min(8, n_out) && groups_fit(block, 2 * K.groups) &&
               2 * K.groups * count <= (long long)resident * block)
            K.groups *= 2;
    K.tile = block / K.groups;
    K.outF = dF ? out_F : tF;
    K.outFc = out_Fc ? (dFc ? out_Fc : tFc) : nullptr;
    K.outG = out_G ? (dG ? out_G : tG) : nullptr;
    K.store_first_g = first;
    CK(launch_bound(kernel_mode(p, true), K, grid, block, smem_bytes(p, block, fs), s));
    p->launches += 1;
    if (!dF) CK(cudaMemcpyAsync(out_F, tF, fb, cudaMemcpyDeviceToHost, s));
    if (out_Fc && !dFc) CK(cudaMemcpyAsync(out_Fc, tFc, fb, cudaMemcpyDeviceToHost, s));
    if (out_G && !dG) CK(cudaMemcpyAsync(out_G, tG, gb, cudaMemcpyDeviceToHost, s));
    if (tF) CK(cudaFreeAsync(tF, s));
    if (tFc) CK(cudaFreeAsync(tFc, s));
    if (tG) CK(cudaFreeAsync(tG, s));
    // the counter copy reads the stack variable first_u: wait before returning
    CK(cudaStreamSynchronize(s));
    return IVB_OK;
}

extern "C" ivb_status ivb_point_grad(ivb_problem* p, int64_t n_points, const double* x, double* out_f,
                                     double* out_grad, void* cuda_stream) {
    if (!p) return fail(nullptr, IVB_EINVAL, "problem handle is NULL");
    p->err.clear();
    if (n_points < 1 || !x || !out_f) return fail(p, IVB_EINVAL, "n_points >= 1, x and out_f are required");
    cudaStream_t s = (cudaStream_t)cuda_stream;
    const int n = p->n, n_out = p->n_out;
    const bool dx = is_device_ptr(x), df = is_device_ptr(out_f), dg = out_grad && is_device_ptr(out_grad);
    const size_t xb = (size_t)n_points * n * sizeof(double), fb = (size_t)n_points * n_out * sizeof(double),
                 gb = fb * n;
    double *tx = nullptr, *tf = nullptr, *tg = nullptr;
    if (!dx) { CK(cudaMallocAsync(&tx, xb, s)); CK(cudaMemcpyAsync(tx, x, xb, cudaMemcpyHostToDevice, s)); }
    if (!df) CK(cudaMallocAsync(&tf, fb, s));
    if (out_grad && !dg) CK(cudaMallocAsync(&tg, gb, s));
    const int units = p->point_units, block = 64;   // small blocks spread few points evenly
    const int grid = (int)std::min<long long>((n_points + block - 1) / block, (long long)p->sm_count * 16);
    const size_t need = (size_t)grid * block * units * sizeof(double);
    if (need > p->pframe_bytes) {
        if (p->d_pframe) CK(cudaFree(p->d_pframe));
        p->d_pframe = nullptr;
        p->pframe_bytes = 0;
        CK(cudaMalloc(&p->d_pframe, need));
        p->pframe_bytes = need;
    }
    CK(launch_point_grad(p->d_prog, n, n_out, units, n_points, dx ? x : tx, df ? out_f : tf,
                         out_grad ? (dg ? out_grad : tg) : nullptr, p->d_pframe, grid, block, s));
    p->launches += 1;
    if (!df) CK(cudaMemcpyAsync(out_f, tf, fb, cudaMemcpyDeviceToHost, s));
    if (out_grad && !dg) CK(cudaMemcpyAsync(out_grad, tg, gb, cudaMemcpyDeviceToHost, s));
    if (tx) CK(cudaFreeAsync(tx, s));
    if (tf) CK(cudaFreeAsync(tf, s));
    if (tg) CK(cudaFreeAsync(tg, s));
    if (!dx || !df || (out_grad && !dg)) CK(cudaStreamSynchronize(s));
    return IVB_OK;
}

extern "C" ivb_status ivb_pick_splits(int32_t n, const double* box, const double* ref_widths, int64_t target,
                                      int32_t strategy, int32_t* out) {
    if (n < 1 || n > IVB_MAX_VARS || !box || !out || target < 1)
        return fail(nullptr, IVB_EINVAL, "pick_splits: n in [1,32], box, out and target >= 1 required");
    if (strategy < 0 || strategy > 2) return fail(nullptr, IVB_EINVAL, "pick_splits: unknown strategy");
    double w[IVB_MAX_VARS];
    for (int i = 0; i < n; ++i) {
        const double wi = box[2 * i + 1] - box[2 * i];
        w[i] = ref_widths ? (ref_widths[i] > 0 ? wi / ref_widths[i] : 0.0) : wi;
    }
    if (strategy == IVB_SPLIT_LARGEST) {
        int wi = 0;
        for (int i = 1; i < n; ++i) if (w[i] > w[wi]) wi = i;
        for (int i = 0; i < n; ++i) out[i] = 1;
        out[wi] = (int32_t)std::min<int64_t>(target, 2147483647);
        return IVB_OK;
    }
    // largest N with N^n <= target
    int64_t N = 1;
    for (;;) {
        const int64_t M = N + 1;
        int64_t prod = 1;
        bool over = false;
        for (int i = 0; i < n && !over; ++i) {
            if (prod > target / M) over = true;
            else prod *= M;
        }
        if (over || prod > target) break;
        N = M;
    }
    for (int i = 0; i < n; ++i) out[i] = (int32_t)N;
    if (strategy == IVB_SPLIT_ADAPTIVE) {
        int64_t prod = 1;
        for (int i = 0; i < n; ++i) prod *= out[i];
        for (;;) {
            int best = -1;
            double bv = -1.0;
            for (int i = 0; i < n; ++i) {
                const int64_t rest = prod / out[i];
                if (rest > target / (out[i] + 1)) continue;
                if (rest * (out[i] + 1) > target) continue;
                const double v = w[i] / out[i];
                if (v > bv) { bv = v; best = i; }
            }
            if (best < 0) break;
            prod = (prod / out[best]) * (out[best] + 1);
            out[best] += 1;
        }
    }
    return IVB_OK;
}

extern "C" ivb_status ivb_get_tuning(ivb_problem* p, int32_t* block_threads, int32_t* blocks_per_sm, int32_t* tile,
                                     int32_t* frame_in_shared) {
    if (!p) return fail(nullptr, IVB_EINVAL, "problem handle is NULL");
    if (block_threads) *block_threads = p->block;
    if (blocks_per_sm) *blocks_per_sm = p->bps;
    if (tile) *tile = p->tile;
    if (frame_in_shared) *frame_in_shared = p->frame_smem;
    return IVB_OK;
}

extern "C" ivb_status ivb_get_tuning_ex(ivb_problem* p, ivb_tuning* t) {
    if (!p || !t) return fail(p, IVB_EINVAL, "problem handle and result are required");
    t->block_threads = p->block;
    t->blocks_per_sm = p->bps;
    t->tile = p->tile;
    t->frame_in_shared = p->frame_smem;
    t->threads_per_subdomain = p->tpsub;
    t->chunk_sync = p->chunk_sync ? 1 : 0;
    t->kernel = reduce_jit(p) ? (p->jit.state_units > 0 ? 2 : 1) : 0;
    t->subdomains_per_pass = pass_size(p, p->block, p->tpsub);
    t->candidates = p->tune_candidates;
    t->best_ms = p->tune_best_ms;
    t->worst_ms = p->tune_worst_ms;
    return IVB_OK;
}

extern "C" ivb_status ivb_get_specialization(ivb_problem* p, int32_t* active, int32_t* registers,
                                             int32_t* local_bytes, double* compile_seconds, int32_t* emulate) {
    if (!p) return fail(nullptr, IVB_EINVAL, "problem handle is NULL");
    if (active) *active = use_jit(p) ? 1 : 0;
    if (emulate) *emulate = use_jit(p) ? p->jit.emulate : 0;
    if (registers) *registers = p->jit.regs;
    if (local_bytes) *local_bytes = p->jit.local_bytes;
    if (compile_seconds) *compile_seconds = p->jit.compile_seconds;
    return IVB_OK;
}

extern "C" ivb_status ivb_get_segmentation(ivb_problem* p, int32_t* state_units, int32_t* chunks,
                                           int64_t* state_loads, int64_t* state_stores, int64_t* recomputed,
                                           int32_t* recompute, int32_t* ilp) {
    if (!p) return fail(nullptr, IVB_EINVAL, "problem handle is NULL");
    const bool seg = use_jit(p) && p->jit.state_units > 0;
    if (state_units) *state_units = seg ? p->jit.state_units : 0;
    if (chunks) *chunks = seg ? p->jit.chunks : 0;
    if (state_loads) *state_loads = seg ? p->jit.state_loads : 0;
    if (state_stores) *state_stores = seg ? p->jit.state_stores : 0;
    if (recomputed) *recomputed = seg ? p->jit.recomputed : 0;
    if (recompute) *recompute = seg ? p->jit.recompute : 0;
    if (ilp) *ilp = seg ? p->jit.ilp : 0;
    return IVB_OK;
}

extern "C" ivb_status ivb_specialize_compile(const ivb_tape* tape, int32_t grad_mode, int32_t compact,
                                             int32_t* registers, int32_t* spill_bytes, double* seconds) {
    std::string e = validate_tape(tape);
    if (!e.empty()) return fail(nullptr, IVB_ETAPE, e);
    if (grad_mode != IVB_GRAD_FORWARD && grad_mode != IVB_GRAD_ADJOINT)
        return fail(nullptr, IVB_EINVAL, "grad_mode must be IVB_GRAD_FORWARD or IVB_GRAD_ADJOINT");
    HostProgram P;
    std::vector<Ins> ins;
    std::vector<RIns> rins;
    std::vector<double> consts;
    e = compile_tape(tape, P, ins, rins, consts);
    if (!e.empty()) return fail(nullptr, IVB_ENOTSUP, e);
    const int mode = grad_mode == IVB_GRAD_ADJOINT ? KM_ADJ_REDUCE : KM_FWD_REDUCE;
    std::vector<char> cubin;
    std::string tables;
    int regs = 0, spill = 0;
    if (compact == 3 || compact == 4) {
        if (grad_mode != IVB_GRAD_ADJOINT)
            return fail(nullptr, IVB_EINVAL, "the segmented kernel needs grad_mode IVB_GRAD_ADJOINT");
        ivb_options o;
        ivb_options_default(&o);
        if (compact == 4) o.seg_ilp = 2;
        const SegPolicy pol = seg_policy(o, P);
        const SegSource src = jit_seg_source(P, ins, rins, consts, seg_block_max(pol.max_regs),
                                             compact == 4 ? 15 : kJitDefaultEmulate, 0, pol);
        e = jit_seg_compile(src, pol.max_regs, cubin, tables, seconds, &regs, &spill);
    } else {
        const std::string src =
            jit_source(P, ins, rins, consts, mode, kJitBlockMax, kJitMinBlocks, kJitDefaultEmulate, compact != 0, 0);
        e = jit_compile(src, cubin, tables, seconds, &regs, &spill);
    }
    if (!e.empty()) return fail(nullptr, IVB_ENOTSUP, e);
    if (registers) *registers = regs;
    if (spill_bytes) *spill_bytes = spill;
    return IVB_OK;
}

extern "C" ivb_status ivb_eval_op(int32_t opcode, int64_t n, const double* x, const double* y, double* r,
                                  void* cuda_stream) {
    if (n < 0 || !x || !r) return fail(nullptr, IVB_EINVAL, "ivb_eval_op: x and r are required");
    const bool binary = opcode == IVB_OP_ADD || opcode == IVB_OP_SUB || opcode == IVB_OP_MUL || opcode == IVB_OP_DIV ||
                        opcode == IVB_EVAL_EMU_ADD || opcode == IVB_EVAL_EMU_SUB || opcode == IVB_EVAL_EMU_MUL ||
                        opcode == IVB_EVAL_FMA;
    const bool unary = opcode == IVB_OP_SQR || opcode == IVB_OP_SQRT || opcode == IVB_OP_EXP || opcode == IVB_OP_LOG ||
                       opcode == IVB_OP_NEG || opcode == IVB_EVAL_RECIP || opcode == IVB_EVAL_EMU_SQR;
    if (!binary && !unary) return fail(nullptr, IVB_EINVAL, "ivb_eval_op: unknown opcode");
    if (binary && !y) return fail(nullptr, IVB_EINVAL, "ivb_eval_op: binary operation needs y");
    if (n == 0) return IVB_OK;
    cudaError_t e = init_math_tables();
    if (e == cudaSuccess) e = launch_eval_op(opcode, n, x, binary ? y : nullptr, r, (cudaStream_t)cuda_stream);
    if (e != cudaSuccess) return fail(nullptr, IVB_ECUDA, std::string("ivb_eval_op: ") + cudaGetErrorString(e));
    return IVB_OK;
}

extern "C" ivb_status ivb_op_counts(const ivb_problem* p, int64_t counts[IVB_CNT_N]) {
    if (!p || !counts) return IVB_EINVAL;
    const bool adj = p->opt.grad_mode == IVB_GRAD_ADJOINT;
    const int64_t* c = p->opt.form == IVB_FORM_NIE ? (adj ? p->P.cnt_nie_adj : p->P.cnt_nie_fwd)
                                                   : (adj ? p->P.cnt_adj : p->P.cnt_fwd);
    for (int i = 0; i < IVB_CNT_N; ++i) counts[i] = c[i];
    return IVB_OK;
}

extern "C" int64_t ivb_launch_count(const ivb_problem* p) { return p ? p->launches : 0; }

extern "C" const char* ivb_last_error(const ivb_problem* p) {
    return p ? p->err.c_str() : g_create_error.c_str();
}

extern "C" void ivb_destroy(ivb_problem* p) {
    if (!p) return;
    drop_graphs(p);
    if (p->cap_stream) cudaStreamDestroy(p->cap_stream);
    if (p->queue_free) { cudaEventSynchronize(p->queue_free); cudaEventDestroy(p->queue_free); }
    cudaFree(p->d_prog);
    cudaFree(p->d_xins);
    cudaFree(p->d_xrins);
    cudaFree(p->d_tan_mask);
    cudaFree(p->d_pins);
    cudaFree(p->d_prins);
    cudaFree(p->d_consts);
    cudaFree(p->d_out_kind);
    cudaFree(p->d_queue);
    if (p->h_queue) cudaFreeHost(p->h_queue);
    cudaFree(p->d_keys);
    cudaFree(p->d_counter);
    cudaFree(p->d_out);
    for (ivb_problem::Pinned* P : {&p->h_in, &p->h_out, &p->h_bnb[0], &p->h_bnb[1]})
        if (P->p) cudaFreeHost(P->p);
    cudaFree(p->d_frame);
    cudaFree(p->d_pframe);
    jit_unload(p->jit);
    delete p;
}
