// capi.cu -- host runtime behind the C ABI of include/mpm.h: device buffers,
// particle load (with the stable block sort of the fused pipeline), tool pose
// streams, CUDA-graph replay of sub-step sequences, readout and inspection.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <utility>
#include <vector>

#include "../../include/mpm.h"
#include "common.cuh"
#include "launch.h"
#include "rotation.h"

using namespace gbmpm;

namespace {

thread_local std::string g_last_error;

mpm_status fail(mpm_status st, const char *fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_last_error = buf;
    return st;
}

#define CK(call)                                                                                    \
    do {                                                                                            \
        cudaError_t e_ = (call);                                                                    \
        if (e_ != cudaSuccess) return fail(MPM_ERR_CUDA, "%s: %s", #call, cudaGetErrorString(e_)); \
    } while (0)


struct HostTool {
    int kind = MPM_TOOL_NONE;
    int field = -1;                       // MPM_TOOL_SAMPLED: index into mpm_handle::fields
    double dims[3] = {0, 0, 0};
    double cur[6] = {0, 0, 0, 0, 0, 0};   // pose at the end of the last sub-step taken
    double tgt[6] = {0, 0, 0, 0, 0, 0};   // pose at the end of the next call
};

struct Alloc {
    void *p;
    size_t bytes;
};

// A sampled distance field registered with mpm_add_sampled_field.
struct HostField {
    const float *d = nullptr;   // res^3 samples in handle-owned device memory
    int res = 0;
    double origin[3] = {0, 0, 0};
    double h = 0;
};

// A recorded differentiable rollout (mpm_tape_record) for mpm_tape_backward.
// A state image holds one split-pipeline particle state: xi, f0, f1, vc0,
// vc1, vc2 (4 n floats each) then f2 (n floats, padded to a multiple of 4).
struct Tape {
    bool valid = false;
    bool settled = false;             // its launches are known to have run to their end
    int nsub = 0, ck = 0, ntools = 0;
    int64_t n = 0;
    size_t image = 0;                 // floats per state image
    size_t cap_ckpt = 0, cap_seg = 0, cap_frames = 0, cap_red = 0, cap_grid = 0, cap_vel = 0, cap_abar = 0;
    float *ckpt = nullptr;            // checkpoint images, one per ck sub-steps
    float *seg = nullptr;             // ck images of the segment being reversed
    float4 *seg_grid = nullptr;       // ck grids (m, mv) as the grid operation read them
    float4 *seg_vel = nullptr;        // ck grids (m, v) the grid operation wrote
    float4 *gv = nullptr;             // scratch grid of the recorded forward pass
    float4 *gbar = nullptr;           // grid adjoint
    float *abar = nullptr;            // particle adjoint: x (3n), v (3n), C (9n), F (9n)
    ToolFrame *frames = nullptr;      // nsub x ntools (device)
    double *red = nullptr;            // dL/dmu, dL/dlam, then nsub x ntools x 18 frame adjoints
    std::vector<double> pose_init;    // ntools x 6
    std::vector<double> poses;        // nsub x ntools x 6
    double E = 0, nu = 0;
    EnvParams mat{};                  // the material and tool count it was recorded with
    EnvParams *d_mat = nullptr;       // and their device copy, where the handle's have changed since
    // fused pipeline: checkpoints are particle-id-ordered images (x, v, F, C:
    // 24 floats per particle); the segment being reversed is replayed with
    // recording sub-steps, each keeping its input particles by block and the
    // grid it read
    bool fused = false;
    float *final_img = nullptr;       // the state after the rollout (restored after the reverse pass)
    size_t cap_final = 0, cap_rs = 0, cap_rsg = 0, cap_rsb = 0, cap_gb = 0;
    float *rs = nullptr;              // nbuf x ck x rs_floats(n): one recorded sub-step's particles
    float4 *rs_grid = nullptr;        // nbuf x ck x 2 nn: the grid each recorded sub-step read, and its velocities
    uint32_t *rs_blk = nullptr;       // ck x (2 nblocks block ranges + nblocks work list + 4 counters)
    float4 *gb2 = nullptr;            // second grid adjoint buffer
    // per grid block: a stamp, and two lists ([count, block ...]) of the blocks
    // a reverse sub-step touches, for the current and the later sub-step
    uint32_t *touch = nullptr;
    size_t cap_touch = 0;
    uint32_t touch_sv = 0;
    double *lame_part = nullptr;      // per CTA of the reverse sub-step: dL/dmu, dL/dlambda
    size_t cap_lame = 0;
    float4 *lp = nullptr;             // 2 x 3 n: state adjoints by position within a segment
    size_t cap_lp = 0;
    bool last_recorded = false;       // the record buffers hold the last segment (from the forward pass)
    // record buffers: one per segment where they fit (kept_record), so that nothing
    // is replayed; otherwise 2 when there is more than one segment
    int nbuf = 1;
    uint32_t end_step = 0;            // h->step at the rollout's end
};

}  // namespace

namespace gbmpm {
void set_last_error(const char *msg) { g_last_error = msg ? msg : ""; }
}  // namespace gbmpm

struct mpm_handle {
    mpm_config cfg{};
    DevParams P{};
    cudaStream_t stream = nullptr;
    cudaStream_t cap_stream = nullptr;
    mpm_alloc_fn alloc_fn = nullptr;
    mpm_free_fn free_fn = nullptr;
    void *alloc_ctx = nullptr;
    std::vector<Alloc> allocs;
    int device = 0, num_sms = 0, fused_grid = 0, elem_grid = 0;
    int kernel_config = 0;          // the fused sub-step's configuration in use
    bool config_set = false;        // by the caller or the autotuner; otherwise by choose_config at each load
    int tuned = 0;                  // mpm_autotune's best where a load's own choice was faster still
    // a load chose 512 threads by the particles' volume, for as long as they use few
    // blocks; or it chose those or 2 CTAs of 256 per SM, for as long as they use not many
    // more than it estimated (adapt_config)
    bool few_blocks = false, by_volume = false;
    uint32_t est_blocks = 0;
    uint32_t load_step = 0;         // the load's sub-step index
    // CTAs by the volume; CTAs of the configurations for more blocks
    int few_ctas = 0, many_grid = 0, default_grid = 0;
    int n_envs = 1;
    int sub_chunk = 512;        // sub-steps per captured graph / frame upload
    int tstride = 0;            // tool frames per environment in the uploaded table
    uint32_t nbe = 0;           // blocks per environment
    uint32_t nblocks = 0, chunk_cap = 0;   // over all environments
    // run lists (fb.runs while a load's configuration and particles need them), their
    // entries, and the configurations whose kernels with them are set up
    uint2 *runs = nullptr;
    size_t runs_cap = 0;
    uint32_t runs_configs = 0;
    int64_t n = 0;
    bool loaded = false;
    uint32_t step = 0;          // fused: device sub-step index mirrored on the host
    int64_t taken = 0;
    float particle_volume = 0.f;
    // buffers
    FusedBufs fb{};
    SortScratch sort{};
    float *staging = nullptr;   // 24 floats per particle (AoS x, v, F, C)
    float4 *dense = nullptr;    // n^3 float4, allocated on first inspection
    ToolFrame *d_frames = nullptr;
    // pinned frame staging, two buffers used in turn: a call waits only for the
    // copy out of the buffer it refills (made two uploads earlier), so the host
    // can run a call ahead of the GPU
    ToolFrame *h_frames[2] = {nullptr, nullptr};
    int frames_next = 0;
    uint32_t *h_err = nullptr;       // pinned copy of Ctrl::err
    uint32_t *h_total = nullptr;     // pinned scratch word: triangles of a surface, error bits
    cudaEvent_t ev_err = nullptr, ev_frames[2] = {nullptr, nullptr};
    // the reverse pass's segment replays run on their own stream, one segment
    // ahead of the reverse sub-steps: rp_rec[b] marks record buffer b complete,
    // rp_free[b] its last reader done, rp_go the start of a reverse pass
    cudaStream_t rp_stream = nullptr;
    cudaEvent_t rp_rec[2] = {nullptr, nullptr}, rp_free[2] = {nullptr, nullptr}, rp_go = nullptr;
    bool err_pending = false;
    std::vector<HostTool> tools;         // n_envs x MPM_MAX_TOOLS
    std::vector<HostField> fields;       // sampled distance fields, shared by every environment
    // per-environment material
    std::vector<double> env_E, env_nu, env_rho, env_vol;
    std::vector<EnvParams> envp_host;
    std::vector<uint32_t> env_off;       // n_envs + 1 particle offsets
    EnvParams *d_envp = nullptr;
    uint32_t *d_env_off = nullptr;
    bool envp_dirty = true;
    std::map<std::pair<int, int>, cudaGraphExec_t> graphs;
    int rev_grid = 0, rec_grid = 0;   // CTAs of the reverse and recording sub-steps
    bool use_graphs = true;
    Tape tape;
    // asynchronous readback: two staging buffers (24 floats per particle), a
    // copy stream, and per buffer the events "gathered" and "copied"
    float *rb_stage[2] = {nullptr, nullptr};
    size_t rb_cap = 0;
    cudaStream_t rb_stream = nullptr;
    cudaEvent_t rb_gathered[2] = {nullptr, nullptr}, rb_copied[2] = {nullptr, nullptr};
    int rb_next = 0;
    bool rb_used[2] = {false, false};
    // autotuner snapshot (24 floats per particle), reused by later calls
    float *tune_snap = nullptr;
    size_t tune_cap = 0;
    // surface extraction scratch
    SurfaceScratch surf{};
    float *surf_tri = nullptr;
    size_t surf_tri_cap = 0;
};

namespace {

mpm_status dalloc(mpm_handle *h, void **out, size_t bytes) {
    bytes = (bytes + 255) & ~size_t(255);
    if (bytes == 0) bytes = 256;
    void *p = nullptr;
    if (h->alloc_fn) {
        p = h->alloc_fn(bytes, (void *)h->stream, h->alloc_ctx);
        if (!p) return fail(MPM_ERR_ALLOC, "allocator callback returned NULL for %zu bytes", bytes);
    } else {
        cudaError_t e = cudaMalloc(&p, bytes);
        if (e != cudaSuccess) return fail(MPM_ERR_ALLOC, "cudaMalloc(%zu): %s", bytes, cudaGetErrorString(e));
    }
    h->allocs.push_back({p, bytes});
    *out = p;
    return MPM_OK;
}

template <typename T>
mpm_status dalloc_t(mpm_handle *h, T **out, size_t count) {
    void *p = nullptr;
    mpm_status st = dalloc(h, &p, count * sizeof(T));
    *out = static_cast<T *>(p);
    return st;
}

// k buffers of `count` elements: one request up to 64 MB (a new handle at 64^3 costs
// 0.2 ms less), or one each, as a caller's allocator may have no piece for all (the
// grids take 2.1 GB each at 512^3, the inboxes 3.7).
template <typename T>
mpm_status dalloc_each(mpm_handle *h, T **out, int k, size_t count) {
    mpm_status st = MPM_OK;
    if (k * count * sizeof(T) <= (size_t)64 << 20) {
        st = dalloc_t(h, &out[0], k * count);
        for (int i = 1; i < k; ++i) out[i] = out[0] + i * count;
        return st;
    }
    for (int i = 0; i < k && st == MPM_OK; ++i) st = dalloc_t(h, &out[i], count);
    return st;
}

// Give one buffer back before the handle ends; no work that uses it may be left.
template <typename T>
void dfree(mpm_handle *h, T **buf, size_t *cap) {
    for (size_t i = 0; i < h->allocs.size(); ++i) {
        if (h->allocs[i].p != *buf) continue;
        if (h->alloc_fn) h->free_fn(*buf, (void *)h->stream, h->alloc_ctx);
        else cudaFree(*buf);
        h->allocs.erase(h->allocs.begin() + (ptrdiff_t)i);
        break;
    }
    *buf = nullptr;
    *cap = 0;
}

void release_all(mpm_handle *h) {
    cudaStreamSynchronize(h->stream);
    if (h->rb_stream) {
        cudaStreamSynchronize(h->rb_stream);
        cudaStreamDestroy(h->rb_stream);
        h->rb_stream = nullptr;
    }
    for (int b = 0; b < 2; ++b) {
        if (h->rb_gathered[b]) cudaEventDestroy(h->rb_gathered[b]);
        if (h->rb_copied[b]) cudaEventDestroy(h->rb_copied[b]);
        h->rb_gathered[b] = h->rb_copied[b] = nullptr;
    }
    for (auto &g : h->graphs) cudaGraphExecDestroy(g.second);
    h->graphs.clear();
    for (auto &a : h->allocs) {
        if (h->alloc_fn) {
            if (h->free_fn) h->free_fn(a.p, (void *)h->stream, h->alloc_ctx);
        } else {
            cudaFree(a.p);
        }
    }
    h->allocs.clear();
    for (int b = 0; b < 2; ++b) {
        if (h->h_frames[b]) cudaFreeHost(h->h_frames[b]);
        if (h->ev_frames[b]) cudaEventDestroy(h->ev_frames[b]);
        h->h_frames[b] = nullptr;
        h->ev_frames[b] = nullptr;
    }
    if (h->rp_stream) {
        cudaStreamSynchronize(h->rp_stream);
        cudaStreamDestroy(h->rp_stream);
        h->rp_stream = nullptr;
    }
    for (int b = 0; b < 2; ++b) {
        if (h->rp_rec[b]) cudaEventDestroy(h->rp_rec[b]);
        if (h->rp_free[b]) cudaEventDestroy(h->rp_free[b]);
        h->rp_rec[b] = h->rp_free[b] = nullptr;
    }
    if (h->rp_go) cudaEventDestroy(h->rp_go);
    h->rp_go = nullptr;
    if (h->h_err) cudaFreeHost(h->h_err);
    if (h->ev_err) cudaEventDestroy(h->ev_err);
    if (h->cap_stream) cudaStreamDestroy(h->cap_stream);
    h->h_err = nullptr;
}

mpm_status status_of(uint32_t err) {
    if (err & kErrNumeric) return fail(MPM_ERR_NUMERIC, "device: non-finite state or det F <= 0");
    if (err & kErrDomain) return fail(MPM_ERR_DOMAIN, "device: a particle stencil left the grid (clamped)");
    if (err & kErrCfl) return fail(MPM_ERR_CFL, "device: a particle moved more than one block in a sub-step");
    if (err & kErrStall) return fail(MPM_ERR_TIMEOUT, "device: the wait between two sub-steps ran out");
    if (err & kErrCapacity) return fail(MPM_ERR_CAPACITY, "device: run-table or particle-count capacity exceeded");
    return MPM_OK;
}

bool is_fused(const mpm_handle *h) { return h->cfg.pipeline == MPM_PIPELINE_FUSED; }

// Device sub-step index for buffer selection.
int cur_par(const mpm_handle *h) { return (int)(h->step & 1u); }
int cur_m3(const mpm_handle *h) { return (int)(h->step % 3u); }

const PState &cur_state(const mpm_handle *h) { return is_fused(h) ? h->fb.P[cur_par(h)] : h->fb.P[0]; }

// Highest active tool slot + 1 over all environments.
int tool_stride(const mpm_handle *h) {
    int ts = 0;
    for (int e = 0; e < h->n_envs; ++e)
        for (int t = 0; t < MPM_MAX_TOOLS; ++t)
            if (h->tools[(size_t)e * MPM_MAX_TOOLS + t].kind != MPM_TOOL_NONE) ts = std::max(ts, t + 1);
    return ts;
}

// Tool frames of nsub sub-steps of a call that moves every tool from its
// current pose to its target uniformly over `total` sub-steps, starting at
// sub-step `first` of the call.  Layout: [sub-step][environment][tool slot],
// tstride slots per environment.
void fill_frames(mpm_handle *h, int first, int nsub, int total, int tstride, ToolFrame *out) {
    const double span = (double)total * (double)h->cfg.dt;
    for (int e = 0; e < h->n_envs; ++e)
        for (int t = 0; t < tstride; ++t) {
            const HostTool &tl = h->tools[(size_t)e * MPM_MAX_TOOLS + t];
            const HostField *fd = tl.kind == MPM_TOOL_SAMPLED ? &h->fields[(size_t)tl.field] : nullptr;
            double reach = 0.0;
            if (tl.kind == MPM_TOOL_CAPSULE) {
                reach = tl.dims[0] + tl.dims[1];
            } else if (tl.kind == MPM_TOOL_BOX) {
                reach = std::sqrt(tl.dims[0] * tl.dims[0] + tl.dims[1] * tl.dims[1] + tl.dims[2] * tl.dims[2]);
            } else if (fd) {   // farthest corner of the sampled volume from the tool origin
                for (int c = 0; c < 8; ++c) {
                    double r2 = 0.0;
                    for (int a = 0; a < 3; ++a) {
                        const double q = fd->origin[a] + ((c >> a) & 1 ? fd->res * fd->h : 0.0);
                        r2 += q * q;
                    }
                    reach = std::max(reach, std::sqrt(r2));
                }
            }
            reach += std::max(0.0, (double)h->cfg.theta);
            reach = reach * 1.001 + 1e-6;
            const CallMotion<double> motion = call_motion(tl.cur, tl.tgt);
            for (int k = 0; k < nsub; ++k) {
                const double s = (double)(first + k + 1) / (double)total;
                ToolFrame &f = out[((size_t)k * h->n_envs + e) * tstride + t];
                std::memset(&f, 0, sizeof f);
                f.kind = tl.kind;
                if (tl.kind == MPM_TOOL_NONE) continue;
                double R[9], T[3], u[3], w[3];
                call_frame(motion, tl.cur, tl.tgt, s, span, R, T, u, w);
                for (int i = 0; i < 9; ++i) f.R[i] = (float)R[i];
                for (int a = 0; a < 3; ++a) {
                    f.T[a] = (float)T[a];
                    f.u[a] = (float)u[a];
                    f.w[a] = (float)w[a];
                    f.dims[a] = (float)(fd ? fd->origin[a] : tl.dims[a]);
                }
                if (fd) {
                    f.res = fd->res;
                    f.inv_h = (float)(1.0 / fd->h);
                    f.sdf = fd->d;
                }
                f.reach2 = (float)(reach * reach);
            }
        }
}

// Per-environment material table and tool counts to the device (when changed).
mpm_status upload_env_params(mpm_handle *h) {
    const int ts = tool_stride(h);
    for (int e = 0; e < h->n_envs; ++e) {
        int nt = 0;
        for (int t = 0; t < MPM_MAX_TOOLS; ++t)
            if (h->tools[(size_t)e * MPM_MAX_TOOLS + t].kind != MPM_TOOL_NONE) nt = t + 1;
        EnvParams &ep = h->envp_host[e];
        const double E = h->env_E[e], nu = h->env_nu[e];   // Eq. 6
        ep.mu = (float)(E / (2.0 * (1.0 + nu)));
        ep.lam = (float)(E * nu / ((1.0 + nu) * (1.0 - 2.0 * nu)));
        ep.mass = (float)(h->env_rho[e] * h->env_vol[e]);
        ep.stress_k = (float)((double)h->cfg.dt * h->env_vol[e] * 4.0 * (double)h->P.inv_dx * h->P.inv_dx);
        ep.ntools = std::min(nt, ts);
    }
    if (ts != h->tstride || h->envp_dirty) {
        CK(cudaStreamSynchronize(h->stream));   // no kernel still reads the old table
        CK(cudaMemcpy(h->d_envp, h->envp_host.data(), sizeof(EnvParams) * h->n_envs, cudaMemcpyHostToDevice));
        h->envp_dirty = false;
    }
    h->tstride = ts;
    h->P.tstride = ts;
    return MPM_OK;
}

// Upload frames for sub-steps [first, first+nsub) of a call of `total`.
mpm_status upload_frames(mpm_handle *h, int first, int nsub, int total) {
    // tool counts can change between calls: refresh the environment table
    mpm_status st = upload_env_params(h);
    if (st != MPM_OK) return st;
    // this staging buffer may still feed the copy of two uploads ago
    const int fb = h->frames_next;
    h->frames_next ^= 1;
    CK(cudaEventSynchronize(h->ev_frames[fb]));
    if (h->tstride > 0) {
        fill_frames(h, first, nsub, total, h->tstride, h->h_frames[fb]);
        CK(cudaMemcpyAsync(h->d_frames, h->h_frames[fb], sizeof(ToolFrame) * (size_t)nsub * h->n_envs * h->tstride,
                           cudaMemcpyHostToDevice, h->stream));
    }
    CK(cudaEventRecord(h->ev_frames[fb], h->stream));
    return MPM_OK;
}

mpm_status poll_error(mpm_handle *h, bool wait) {
    if (!h->err_pending) return MPM_OK;
    if (wait) {
        CK(cudaEventSynchronize(h->ev_err));
    } else {
        cudaError_t q = cudaEventQuery(h->ev_err);
        if (q == cudaErrorNotReady) return MPM_OK;
        if (q != cudaSuccess) return fail(MPM_ERR_CUDA, "cudaEventQuery: %s", cudaGetErrorString(q));
    }
    return status_of(*h->h_err);
}

// A rollout whose recording launches lost one another has records of sub-steps that
// never ran: it must not be reversed.  Waits for the launches, once per rollout.
mpm_status settle_tape(mpm_handle *h) {
    Tape &tp = h->tape;
    if (!tp.valid || tp.settled) return MPM_OK;
    CK(cudaEventSynchronize(h->ev_err));
    tp.settled = true;
    if (*h->h_err & kErrStall) tp.valid = false;
    return MPM_OK;
}

mpm_status enqueue_error_copy(mpm_handle *h) {
    CK(cudaMemcpyAsync(h->h_err, &h->fb.ctrl->err, sizeof(uint32_t), cudaMemcpyDeviceToHost, h->stream));
    CK(cudaEventRecord(h->ev_err, h->stream));
    h->err_pending = true;
    return MPM_OK;
}

// The number of blocks in use that the last finished launch since the load
// reported, or 0.
uint32_t blocks_reported(const mpm_handle *h) {
    const unsigned long long w = *(volatile unsigned long long *)h->fb.host_blocks;
    return (int32_t)((uint32_t)w - h->load_step) > 0 ? (uint32_t)(w >> 32) : 0u;
}

// 512 threads as a load chose them pay off while every block has a CTA.  The volume
// tells the blocks of a body in one piece; particles that lie scattered, or come
// apart, use many more (2,000 strewn over the 32^3 grid: 380 blocks on 32 CTAs, 1,380
// us a frame; with 2 CTAs of 256 threads per SM 300).  By what the last launch
// reported those take over, and give back at half as many; from four blocks per SM on
// 3 CTAs per SM do, until the next load (8,192 strewn over the 64^3 grid, 2,400
// blocks: 5,430 us, 2 per SM 1,070, 3 per SM 940; 30,000 over the 128^3 grid,
// 14,300 blocks: 10,300, 5,750, 4,850).  So they do for a load's 2 CTAs per SM once the
// blocks are four times its estimate (60,000 over the 128^3 grid: 6,790 against 5,700).
constexpr int kConfigMany = MPM_KERNEL_T256_G2_C2;
void adapt_config(mpm_handle *h) {
    const uint32_t blocks = h->by_volume ? blocks_reported(h) : 0u, sms = (uint32_t)h->num_sms;
    if (blocks == 0) return;
    if (blocks > 4 * std::max(sms, h->est_blocks)) {
        h->few_blocks = h->by_volume = false;
        h->kernel_config = MPM_KERNEL_T256_G2;
        h->fused_grid = h->default_grid;
        return;
    }
    if (!h->few_blocks) return;
    const bool many = blocks > (h->kernel_config == kConfigT512 ? sms : sms / 2);
    h->kernel_config = many ? kConfigMany : kConfigT512;
    h->fused_grid = many ? h->many_grid : (int)std::min(sms, std::max((uint32_t)h->few_ctas, blocks));
}

// Issue nsub sub-steps on stream st (used directly and under capture).
mpm_status issue_substeps(mpm_handle *h, int nsub, bool write_vc_last, cudaStream_t st) {
    const DevParams P = h->P;
    const uint32_t n = (uint32_t)h->n;
    if (is_fused(h)) {
        // a load's 512 threads, before any launch has reported the blocks in use: its
        // kernel takes the call up to one block per SM, otherwise the one behind it does
        // (3 us for the one that has nothing to do, in the first call after a load)
        LaunchGate gate;
        const bool unsure = h->few_blocks && !blocks_reported(h);
        if (unsure) {
            gate.most_blocks = (uint32_t)h->num_sms;
            gate.at = h->step;
        }
        launch_fused_steps(P, h->fb, h->d_frames, nsub, write_vc_last, h->fused_grid, h->kernel_config, st, gate);
        if (unsure) {
            gate.most_blocks = LaunchGate::kAny;
            launch_fused_steps(P, h->fb, h->d_frames, nsub, write_vc_last, h->many_grid, kConfigMany, st, gate);
        }
        CK(cudaGetLastError());
        return MPM_OK;
    }
    for (int k = 0; k < nsub; ++k) {
        const ToolFrame *fr = h->d_frames + (size_t)k * h->n_envs * h->tstride;
        CK(cudaMemsetAsync(h->fb.G[0], 0, sizeof(float4) * (size_t)h->P.n * h->P.n * h->P.n, st));
        launch_p2g_scatter(P, h->fb.P[0], h->fb.vc, n, h->fb.G[0], h->fb.ctrl, h->elem_grid, st);
        launch_grid_update_dense(P, h->fb.G[0], fr, h->elem_grid, st);
        launch_g2p_split(P, h->fb.P[0], h->fb.vc, n, h->fb.G[0], h->fb.ctrl, h->elem_grid, st);
    }
    CK(cudaGetLastError());
    return MPM_OK;
}

mpm_status run_chunk(mpm_handle *h, int nsub, bool write_vc_last) {
    // one or two launches need no graph
    if (!h->use_graphs || (is_fused(h) && fused_many_steps(h->kernel_config))) return issue_substeps(h, nsub, write_vc_last, h->stream);
    // graphs are keyed by length, the vc flag, the tool-frame stride and the kernel configuration
    const std::pair<int, int> key(nsub, (write_vc_last ? 1 : 0) | (h->tstride << 1) | (h->kernel_config << 8));
    auto it = h->graphs.find(key);
    if (it == h->graphs.end()) {
        cudaGraph_t g = nullptr;
        CK(cudaStreamBeginCapture(h->cap_stream, cudaStreamCaptureModeThreadLocal));
        mpm_status st = issue_substeps(h, nsub, write_vc_last, h->cap_stream);
        cudaError_t e = cudaStreamEndCapture(h->cap_stream, &g);
        if (st != MPM_OK) {
            if (g) cudaGraphDestroy(g);
            return st;
        }
        if (e != cudaSuccess) return fail(MPM_ERR_CUDA, "cudaStreamEndCapture: %s", cudaGetErrorString(e));
        cudaGraphExec_t ex = nullptr;
        e = cudaGraphInstantiate(&ex, g, 0);
        cudaGraphDestroy(g);
        if (e != cudaSuccess) return fail(MPM_ERR_CUDA, "cudaGraphInstantiate: %s", cudaGetErrorString(e));
        it = h->graphs.emplace(key, ex).first;
    }
    CK(cudaGraphLaunch(it->second, h->stream));
    return MPM_OK;
}

mpm_status check_handle(mpm_handle *h) {
    if (!h) return fail(MPM_ERR_ARG, "NULL handle");
    int dev = -1;
    CK(cudaGetDevice(&dev));
    if (dev != h->device) CK(cudaSetDevice(h->device));
    return MPM_OK;
}

}  // namespace

// =================================================================== ABI

extern "C" {

const char *mpm_last_error(void) { return g_last_error.c_str(); }

mpm_status mpm_create(const mpm_config *cfg, void *cuda_stream, mpm_alloc_fn alloc, mpm_free_fn free_fn, void *ctx,
                      mpm_handle **out) {
    if (!cfg || !out) return fail(MPM_ERR_ARG, "mpm_create: NULL config or output pointer");
    *out = nullptr;
    const int n = cfg->n_grid;
    if (n < 8 || n > 512 || (n & (n - 1)) != 0) return fail(MPM_ERR_ARG, "n_grid must be a power of two in [8, 512]");
    if (cfg->bound < 0 || 2 * cfg->bound >= n) return fail(MPM_ERR_ARG, "bound out of range");
    if (!(cfg->dt > 0.f) || !std::isfinite(cfg->dt)) return fail(MPM_ERR_ARG, "dt must be positive");
    if (!(cfg->E >= 0.f) || !(cfg->nu >= 0.f) || !(cfg->nu < 0.5f)) return fail(MPM_ERR_ARG, "need E >= 0, 0 <= nu < 0.5");
    if (!(cfg->rho > 0.f)) return fail(MPM_ERR_ARG, "rho must be positive");
    if (!(cfg->friction_mu >= 0.f)) return fail(MPM_ERR_ARG, "friction_mu must be >= 0");
    if (!std::isfinite(cfg->theta) || !std::isfinite(cfg->gravity[0]) || !std::isfinite(cfg->gravity[1]) ||
        !std::isfinite(cfg->gravity[2]))
        return fail(MPM_ERR_ARG, "theta and gravity must be finite");
    if (cfg->pipeline != MPM_PIPELINE_FUSED && cfg->pipeline != MPM_PIPELINE_SPLIT)
        return fail(MPM_ERR_ARG, "unknown pipeline %d", cfg->pipeline);
    if (cfg->max_particles < 1 || cfg->max_particles > (int64_t)1 << 30)
        return fail(MPM_ERR_ARG, "max_particles must be in [1, 2^30]");
    const int n_envs = cfg->n_envs < 1 ? 1 : cfg->n_envs;
    if (n_envs > 65536) return fail(MPM_ERR_ARG, "n_envs must be at most 65536");
    if (n_envs > 1 && cfg->pipeline != MPM_PIPELINE_FUSED)
        return fail(MPM_ERR_ARG, "several environments need the fused pipeline");
    if ((uint64_t)n_envs * (uint64_t)(n / 4) * (n / 4) * (n / 4) > (1ull << 26))
        return fail(MPM_ERR_ARG, "n_envs * (n_grid/4)^3 grid blocks exceed 2^26");
    if ((alloc == nullptr) != (free_fn == nullptr)) return fail(MPM_ERR_ARG, "alloc and free callbacks go together");

    mpm_handle *h = new (std::nothrow) mpm_handle();
    if (!h) return fail(MPM_ERR_ALLOC, "host allocation of the handle failed");
    h->cfg = *cfg;
    h->stream = (cudaStream_t)cuda_stream;
    h->alloc_fn = alloc;
    h->free_fn = free_fn;
    h->alloc_ctx = ctx;
    const char *ng = getenv("GBMPM_NO_GRAPHS");
    h->use_graphs = !(ng && ng[0] == '1');
    // looks of the wait between two sub-steps of a launch: a few seconds' worth, or
    // fewer by GBMPM_WAIT_POLLS (which lets a test make the wait run out)
    h->fb.max_polls = 1u << 22;
    const char *wp = getenv("GBMPM_WAIT_POLLS");
    const long polls = wp ? std::strtol(wp, nullptr, 10) : 0;
    if (polls > 0) h->fb.max_polls = (uint32_t)std::min<long>(polls, h->fb.max_polls);

    auto bail = [&](mpm_status st) {
        release_all(h);
        delete h;
        return st;
    };
    cudaError_t e = cudaGetDevice(&h->device);
    if (e != cudaSuccess) return bail(fail(MPM_ERR_CUDA, "cudaGetDevice: %s", cudaGetErrorString(e)));
    e = cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, h->device);
    if (e != cudaSuccess) return bail(fail(MPM_ERR_CUDA, "cudaDeviceGetAttribute: %s", cudaGetErrorString(e)));

    h->n_envs = n_envs;
    h->tools.assign((size_t)n_envs * MPM_MAX_TOOLS, HostTool());
    h->env_E.assign(n_envs, cfg->E);
    h->env_nu.assign(n_envs, cfg->nu);
    h->env_rho.assign(n_envs, cfg->rho);
    h->env_vol.assign(n_envs, 0.0);
    h->envp_host.assign(n_envs, EnvParams{});
    h->env_off.assign(n_envs + 1, 0u);
    h->sub_chunk = std::max(1, std::min(512, 16384 / n_envs));
    DevParams &P = h->P;
    P.n = n;
    P.nb = n / 4;
    while ((4 << P.lnb) < n) ++P.lnb;      // n is a power of two
    P.nbe = (uint32_t)(P.nb * P.nb * P.nb);
    P.n_envs = n_envs;
    P.bound = cfg->bound;
    P.tstride = 0;
    P.dx = 1.0f / (float)n;
    P.inv_dx = (float)n;
    P.dt = cfg->dt;
    P.gx = cfg->gravity[0];
    P.gy = cfg->gravity[1];
    P.gz = cfg->gravity[2];
    P.theta = cfg->theta;
    P.fric = cfg->friction_mu;

    const size_t N = (size_t)cfg->max_particles;
    const size_t nn = (size_t)n * n * n * n_envs;   // grid nodes over all environments
    h->nbe = P.nbe;
    h->nblocks = P.nbe * (uint32_t)n_envs;
    h->chunk_cap = h->nblocks + (uint32_t)(N / kFusedMinThreads) + 1;
    h->fb.nblocks = h->nblocks;
    h->elem_grid = h->num_sms * 8;
    const int occ = fused_step_occupancy(h->kernel_config);
    h->fused_grid = h->default_grid = h->num_sms * std::max(occ, 1);

    mpm_status st;
    const int nbuf = cfg->pipeline == MPM_PIPELINE_FUSED ? 2 : 1;
    // both buffers of an array in one allocation (the second starts on a 256-byte boundary)
    const size_t ps = (N + 63) & ~size_t(63);
    h->fb.pstride = nbuf == 2 ? (uint32_t)ps : 0u;
    h->fb.cstride = h->chunk_cap;
    PState &P0 = h->fb.P[0], &P1 = h->fb.P[1];
    if ((st = dalloc_t(h, &P0.xi, ps * nbuf)) != MPM_OK) return bail(st);
    if ((st = dalloc_t(h, &P0.f0, ps * nbuf)) != MPM_OK) return bail(st);
    if ((st = dalloc_t(h, &P0.f1, ps * nbuf)) != MPM_OK) return bail(st);
    if ((st = dalloc_t(h, &P0.f2, ps * nbuf)) != MPM_OK) return bail(st);
    P1 = {P0.xi + h->fb.pstride, P0.f0 + h->fb.pstride, P0.f1 + h->fb.pstride, P0.f2 + h->fb.pstride};
    if ((st = dalloc_t(h, &h->fb.vc.vc0, N)) != MPM_OK) return bail(st);
    if ((st = dalloc_t(h, &h->fb.vc.vc1, N)) != MPM_OK) return bail(st);
    if ((st = dalloc_t(h, &h->fb.vc.vc2, N)) != MPM_OK) return bail(st);
    const int ngrid = cfg->pipeline == MPM_PIPELINE_FUSED ? 3 : 1;
    if ((st = dalloc_each(h, h->fb.G, ngrid, nn)) != MPM_OK) return bail(st);
    for (int g = ngrid; g < 3; ++g) h->fb.G[g] = h->fb.G[0];
    if ((st = dalloc_t(h, &h->fb.ctrl, 1)) != MPM_OK) return bail(st);
    if ((st = dalloc_t(h, &h->staging, 24 * N)) != MPM_OK) return bail(st);
    if ((st = dalloc_t(h, &h->d_frames, (size_t)h->sub_chunk * n_envs * MPM_MAX_TOOLS)) != MPM_OK) return bail(st);
    if ((st = dalloc_t(h, &h->d_envp, (size_t)n_envs)) != MPM_OK) return bail(st);
    if ((st = dalloc_t(h, &h->d_env_off, (size_t)n_envs + 1)) != MPM_OK) return bail(st);
    P.envp = h->d_envp;
    P.env_off = h->d_env_off;
    if (cfg->pipeline == MPM_PIPELINE_FUSED) {
        const size_t nblk = h->nblocks;
        if ((st = dalloc_t(h, &h->fb.chunks[0], 2 * (size_t)h->chunk_cap)) != MPM_OK) return bail(st);
        if ((st = dalloc_t(h, &h->fb.tabs[0], 2 * nblk)) != MPM_OK) return bail(st);
        if ((st = dalloc_t(h, &h->fb.alist[0], 2 * nblk)) != MPM_OK) return bail(st);
        if ((st = dalloc_each(h, h->fb.inbox, 2, nblk * kInbox)) != MPM_OK) return bail(st);
        h->fb.chunks[1] = h->fb.chunks[0] + h->chunk_cap;
        h->fb.tabs[1] = h->fb.tabs[0] + nblk;
        h->fb.alist[1] = h->fb.alist[0] + nblk;
        for (int b = 0; b < 3; ++b)
            if ((st = dalloc_t(h, &h->fb.clist[b], h->nblocks)) != MPM_OK) return bail(st);
        if ((st = dalloc_t(h, &h->fb.astamp, h->nblocks)) != MPM_OK) return bail(st);
        if ((st = dalloc_t(h, &h->fb.gstamp, h->nblocks)) != MPM_OK) return bail(st);
        if ((st = dalloc_t(h, &h->sort.keys, N)) != MPM_OK) return bail(st);
        if ((st = dalloc_t(h, &h->sort.perm, N)) != MPM_OK) return bail(st);
        if ((st = dalloc_t(h, &h->sort.counts, h->nblocks)) != MPM_OK) return bail(st);
        if ((st = dalloc_t(h, &h->sort.offsets, h->nblocks + 1)) != MPM_OK) return bail(st);
        if ((st = dalloc_t(h, &h->sort.cursor, h->nblocks)) != MPM_OK) return bail(st);
    }
    for (int b = 0; b < 2; ++b) {
        e = cudaMallocHost(&h->h_frames[b], sizeof(ToolFrame) * (size_t)h->sub_chunk * n_envs * MPM_MAX_TOOLS);
        if (e != cudaSuccess) return bail(fail(MPM_ERR_ALLOC, "cudaMallocHost: %s", cudaGetErrorString(e)));
    }
    e = cudaMallocHost(&h->h_err, 4 * sizeof(uint32_t));
    if (e != cudaSuccess) return bail(fail(MPM_ERR_ALLOC, "cudaMallocHost: %s", cudaGetErrorString(e)));
    *h->h_err = 0;
    h->h_total = h->h_err + 1;
    h->fb.host_err = h->h_err;
    h->fb.host_blocks = reinterpret_cast<unsigned long long *>(h->h_err + 2);
    *h->fb.host_blocks = 0;
    if ((e = cudaEventCreateWithFlags(&h->ev_err, cudaEventDisableTiming)) != cudaSuccess ||
        (e = cudaEventCreateWithFlags(&h->ev_frames[0], cudaEventDisableTiming)) != cudaSuccess ||
        (e = cudaEventCreateWithFlags(&h->ev_frames[1], cudaEventDisableTiming)) != cudaSuccess ||
        (e = cudaStreamCreateWithFlags(&h->cap_stream, cudaStreamNonBlocking)) != cudaSuccess)
        return bail(fail(MPM_ERR_CUDA, "event/stream creation: %s", cudaGetErrorString(e)));
    e = cudaEventRecord(h->ev_frames[0], h->stream);
    if (e == cudaSuccess) e = cudaEventRecord(h->ev_frames[1], h->stream);
    if (e == cudaSuccess && h->fb.astamp) e = cudaMemsetAsync(h->fb.astamp, 0, sizeof(uint32_t) * h->nblocks, h->stream);
    if (e == cudaSuccess && h->fb.gstamp) e = cudaMemsetAsync(h->fb.gstamp, 0, sizeof(uint32_t) * h->nblocks, h->stream);
    for (int b = 0; b < 2 && e == cudaSuccess && h->fb.tabs[b]; ++b) {
        e = cudaMemsetAsync(h->fb.tabs[b], 0, sizeof(BlockTab) * h->nblocks, h->stream);
        if (e == cudaSuccess) e = cudaMemsetAsync(h->fb.inbox[b], 0, sizeof(uint4) * h->nblocks * kInbox, h->stream);
    }
    if (e == cudaSuccess) e = cudaMemsetAsync(h->fb.ctrl, 0, sizeof(Ctrl), h->stream);
    if (e != cudaSuccess) return bail(fail(MPM_ERR_CUDA, "initial clears: %s", cudaGetErrorString(e)));
    *out = h;
    return MPM_OK;
}

mpm_status mpm_destroy(mpm_handle *h) {
    if (!h) return fail(MPM_ERR_ARG, "NULL handle");
    cudaSetDevice(h->device);
    release_all(h);
    delete h;
    return MPM_OK;
}

mpm_status mpm_set_stream(mpm_handle *h, void *cuda_stream) {
    mpm_status st = check_handle(h);
    if (st != MPM_OK) return st;
    h->stream = (cudaStream_t)cuda_stream;
    CK(cudaEventRecord(h->ev_frames[0], h->stream));
    CK(cudaEventRecord(h->ev_frames[1], h->stream));
    return MPM_OK;
}

}  // extern "C"

namespace {

mpm_status apply_kernel_config(mpm_handle *h, int config);

// The loaded particles' volume in full 4x4x4 blocks.
double full_blocks(const mpm_handle *h) {
    const double cell = 1.0 / ((double)h->P.n * h->P.n * h->P.n);
    double full = 0.0;
    for (int e = 0; e < h->n_envs; ++e)
        full += (double)(h->env_off[e + 1] - h->env_off[e]) * h->env_vol[e] / (64.0 * cell);
    return full;
}

bool is_sparse(const mpm_handle *h) { return (double)h->n < 6.0 * 64.0 * full_blocks(h); }
double estimated_blocks(const mpm_handle *h) { return full_blocks(h) * (is_sparse(h) ? 2.0 : 1.5); }

static_assert(kConfigT512 == MPM_KERNEL_CONFIGS, "the library's own configuration follows the selectable ones");
// The fused sub-step's configuration for the loaded particles, where the caller
// has set none.  By the number of filled 4x4x4 blocks, estimated as the particles
// over a full block's number (64 cells' worth, from their volume) times 1.5, or
// times 2 for sparse bodies, as the blocks at the surface are filled in part.
// Measured on 152 SMs, us per sub-step under configurations 0, 2, 3, 4 and 5:
// - as long as every block can have a CTA of its own, one block's chain counts, so
//   the largest CTAs that fit (8K cube 21.7, 37, 43, 21.8, 18.1; 50K at 10 per cell
//   17.8, 22.7, 25.6, 14.2, 12.8; 30K slab 17.1, 17.7, 21.4, 13.8, 17.5);
// - with 2 CTAs per SM that holds to 3 estimated blocks per SM, as long as an SM has up
//   to 400 particles.  Slabs on 64^3, us per frame of 25 sub-steps under 2, 3 and 4, at
//   3.2 per cell: 31K 368, 442, 249; 40K 404, 470, 360; 45K 399, 463, 364; 50K (3.2
//   blocks per SM) 407, 478, 380; at 4 per cell: 56K 404, 476, 393; at 5 per cell: 60K
//   417, 453, 413; 65K (430 particles per SM) 423, 454, 430; 72K 421, 465, 443;
// - beyond, sparse blocks waste the fewest threads of the smallest CTAs (200K slab
//   47, 43, 39, 45, 61; 256 environments 1389, 1200, 1150, 1520, 2340), dense ones
//   run from 4 to 5 blocks per CTA on with the most warps (500K at 8 per cell 51.4,
//   59, 61, 50.5, 70; 800K 72.4, 81, 86, 76.3, 106; 1M 94, 105, 109, 100, 138).
int choose_config(const mpm_handle *h) {
    const double sms = h->num_sms, blocks = estimated_blocks(h);
    const bool sparse = is_sparse(h);
    if (blocks <= sms) return kConfigT512;
    if (blocks <= 2.0 * sms || (blocks <= 3.0 * sms && (double)h->n <= 400.0 * sms)) return MPM_KERNEL_T256_G2_C2;
    if (sparse) return blocks <= 4.0 * sms ? MPM_KERNEL_T128_G2 : MPM_KERNEL_T128_G1;
    return blocks <= 9.0 * sms ? MPM_KERNEL_T256_G2_C2 : MPM_KERNEL_T256_G2;
}

// CTAs of 512 threads for the loaded particles: a few for every block (a body may
// spread), not one per SM, as each more arrives at and polls the wait between
// sub-steps (2K patch 104 -> 100 us a call).
int few_ctas(const mpm_handle *h) {
    return std::min(h->num_sms, std::max(32, (int)std::ceil(6.0 * full_blocks(h))));
}

// Where 128-thread CTAs step an environment whose blocks may take in more runs than
// shared memory holds (a 27-block neighbourhood of t particles writes at most
// t / 128 + 27 chunks): the lists in global memory, 8 KB a CTA.
mpm_status ensure_runs(mpm_handle *h) {
    h->fb.runs = nullptr;
    const int config = h->kernel_config;
    if (fused_step_threads(config) >= 256) return MPM_OK;
    uint32_t most = 0;
    for (int e = 0; e < h->n_envs; ++e) most = std::max(most, h->env_off[e + 1] - h->env_off[e]);
    if (most <= (kRunsShared - 27) * 128) return MPM_OK;
    // its kernels opt into their shared memory, once; the grid is that of the others
    if (!(h->runs_configs >> config & 1u)) {
        if (h->num_sms * fused_step_occupancy(config, true) < h->fused_grid)
            return fail(MPM_ERR_ALLOC, "kernel configuration %d with run lists does not fit", config);
        h->runs_configs |= 1u << config;
    }
    const size_t count = (size_t)h->fused_grid * kRunsListed;
    if (h->runs_cap < count) {
        uint2 *runs = nullptr;
        const mpm_status st = dalloc_t(h, &runs, count);
        if (st != MPM_OK) {
            cudaGetLastError();
            return st;
        }
        h->runs = runs;
        h->runs_cap = count;
    }
    h->fb.runs = h->runs;
    return MPM_OK;
}

// Replace the state of every environment: counts[e] particles of environment
// e, stored env-major in x, v, F, C; volumes[e] its particle volume.
mpm_status load_impl(mpm_handle *h, const int64_t *counts, const float *x, const float *v, const float *F,
                     const float *C, const float *volumes, int on_device) {
    int64_t total = 0;
    for (int e = 0; e < h->n_envs; ++e) {
        if (counts[e] < 0) return fail(MPM_ERR_ARG, "negative particle count for environment %d", e);
        if (!(volumes[e] > 0.f) || !std::isfinite(volumes[e]))
            return fail(MPM_ERR_ARG, "particle volume of environment %d must be > 0", e);
        total += counts[e];
    }
    if (total > h->cfg.max_particles)
        return fail(MPM_ERR_ARG, "%lld particles exceed max_particles", (long long)total);
    if (total > 0 && !x) return fail(MPM_ERR_ARG, "x is required");
    const int64_t n = total;
    const size_t N = (size_t)n;
    // inputs in device memory (staging copies for host inputs)
    const float *dx = x, *dv = v, *dF = F, *dC = C;
    if (!on_device && n > 0) {
        float *sx = h->staging, *sv = sx + 3 * N, *sF = sv + 3 * N, *sC = sF + 9 * N;
        CK(cudaMemcpyAsync(sx, x, sizeof(float) * 3 * N, cudaMemcpyHostToDevice, h->stream));
        dx = sx;
        if (v) { CK(cudaMemcpyAsync(sv, v, sizeof(float) * 3 * N, cudaMemcpyHostToDevice, h->stream)); dv = sv; }
        if (F) { CK(cudaMemcpyAsync(sF, F, sizeof(float) * 9 * N, cudaMemcpyHostToDevice, h->stream)); dF = sF; }
        if (C) { CK(cudaMemcpyAsync(sC, C, sizeof(float) * 9 * N, cudaMemcpyHostToDevice, h->stream)); dC = sC; }
    }
    h->particle_volume = volumes[0];
    h->env_off[0] = 0;
    for (int e = 0; e < h->n_envs; ++e) {
        if (h->env_vol[e] != (double)volumes[e]) h->envp_dirty = true;   // the particle mass changes
        h->env_vol[e] = volumes[e];
        h->env_off[e + 1] = h->env_off[e] + (uint32_t)counts[e];
    }
    // graphs captured the old parameters
    for (auto &g : h->graphs) cudaGraphExecDestroy(g.second);
    h->graphs.clear();

    Ctrl c{};
    const uint32_t k0 = h->step + 2;   // fresh stamps: every table entry from before is older
    c.step = k0;
    c.n_particles = (uint32_t)n;
    CK(cudaMemcpyAsync(h->fb.ctrl, &c, sizeof c, cudaMemcpyHostToDevice, h->stream));
    CK(cudaMemcpyAsync(h->d_env_off, h->env_off.data(), sizeof(uint32_t) * (h->n_envs + 1), cudaMemcpyHostToDevice,
                       h->stream));
    // host inputs (possibly pinned, so copied asynchronously) must outlive their
    // copies; c and env_off are pageable, which cudaMemcpyAsync stages at once
    if (!on_device && n > 0) CK(cudaStreamSynchronize(h->stream));
    mpm_status st = upload_env_params(h);
    if (st != MPM_OK) return st;
    h->step = k0;
    h->load_step = k0;
    h->few_blocks = h->by_volume = false;
    h->n = n;
    h->taken = 0;
    if (is_fused(h) && !h->config_set) {
        const int config = choose_config(h);
        if (config != h->kernel_config && (st = apply_kernel_config(h, config)) != MPM_OK) return st;
        h->few_blocks = config == kConfigT512;
        h->by_volume = h->few_blocks || config == kConfigMany;
        h->est_blocks = (uint32_t)std::min(estimated_blocks(h), 1e9);
        if (h->few_blocks) {
            h->fused_grid = h->few_ctas = few_ctas(h);
            if (h->many_grid == 0) h->many_grid = h->num_sms * std::max(fused_step_occupancy(kConfigMany), 1);
            CK(cudaGetLastError());
        }
        // without the lists, 256 threads keep a block's capacity
        if (ensure_runs(h) != MPM_OK && (st = apply_kernel_config(h, MPM_KERNEL_T256_G2_C2)) != MPM_OK) return st;
    } else if (is_fused(h)) {
        if (h->kernel_config == kConfigT512) h->fused_grid = few_ctas(h);     // a trial of the autotuner
        ensure_runs(h);
    }
    const size_t nn = (size_t)h->P.n * h->P.n * h->P.n * h->n_envs;
    if (is_fused(h)) {
        launch_clear_grids(h->fb, nn, h->elem_grid, h->stream);
        CK(cudaMemsetAsync(h->sort.counts, 0, sizeof(uint32_t) * h->nblocks, h->stream));
        launch_block_sort(h->P, dx, (uint32_t)n, h->sort, h->fb.ctrl, h->elem_grid, h->stream);
        const int par = cur_par(h);
        launch_place_sorted(h->P, dx, dv, dF, dC, (uint32_t)n, h->sort, h->fb.P[par], h->fb.vc, h->elem_grid, h->stream);
        launch_init_tables(h->P, h->sort, h->fb, k0, h->elem_grid, h->stream);
        launch_p2g_scatter(h->P, h->fb.P[par], h->fb.vc, (uint32_t)n, h->fb.G[cur_m3(h)], h->fb.ctrl, h->elem_grid,
                           h->stream);
    } else {
        launch_load_identity(dx, dv, dF, dC, (uint32_t)n, h->fb.P[0], h->fb.vc, h->fb.ctrl, h->elem_grid, h->stream);
    }
    CK(cudaGetLastError());
    h->loaded = true;
    if (!on_device) CK(cudaStreamSynchronize(h->stream));
    return enqueue_error_copy(h);
}

mpm_status set_tool_impl(mpm_handle *h, int32_t env, int32_t tool_id, const double pose[6], const float shape[8]) {
    if (env < 0 || env >= h->n_envs) return fail(MPM_ERR_ARG, "environment %d out of range", env);
    if (tool_id < 0 || tool_id >= MPM_MAX_TOOLS) return fail(MPM_ERR_ARG, "tool_id %d out of range", tool_id);
    if (!pose || !shape) return fail(MPM_ERR_ARG, "NULL pose or shape");
    HostTool &t = h->tools[(size_t)env * MPM_MAX_TOOLS + tool_id];
    const int kind = (int)shape[0];
    if (kind == MPM_TOOL_NONE) {
        t = HostTool();
        return MPM_OK;
    }
    if (kind != MPM_TOOL_CAPSULE && kind != MPM_TOOL_BOX && kind != MPM_TOOL_SAMPLED)
        return fail(MPM_ERR_ARG, "unknown tool kind %d", kind);
    for (int i = 0; i < 6; ++i)
        if (!std::isfinite(pose[i])) return fail(MPM_ERR_ARG, "non-finite pose");
    int field = -1;
    if (kind == MPM_TOOL_SAMPLED) {
        if (!(shape[1] >= 0.f) || shape[1] != std::floor(shape[1]) || shape[1] >= (float)h->fields.size())
            return fail(MPM_ERR_ARG, "shape[1] = %g is not a registered sampled field", (double)shape[1]);
        field = (int)shape[1];
    } else {
        for (int i = 1; i < 4; ++i)
            if (!(shape[i] >= 0.f) || !std::isfinite(shape[i]))
                return fail(MPM_ERR_ARG, "shape sizes must be finite and >= 0");
    }
    const bool fresh = t.kind == MPM_TOOL_NONE;
    t.kind = kind;
    t.field = field;
    for (int a = 0; a < 3; ++a) t.dims[a] = kind == MPM_TOOL_SAMPLED ? 0.0 : shape[1 + a];
    for (int i = 0; i < 6; ++i) {
        t.tgt[i] = pose[i];
        if (fresh) t.cur[i] = pose[i];
    }
    return MPM_OK;
}

}  // namespace

extern "C" {

mpm_status mpm_load_particles(mpm_handle *h, int64_t n, const float *x, const float *v, const float *F, const float *C,
                              float particle_volume, int on_device) {
    mpm_status st = check_handle(h);
    if (st != MPM_OK) return st;
    if (h->n_envs != 1) return fail(MPM_ERR_STATE, "a handle with several environments loads with mpm_load_batch");
    if (n < 0 || n > h->cfg.max_particles) return fail(MPM_ERR_ARG, "n = %lld outside [0, max_particles]", (long long)n);
    if ((st = settle_tape(h)) != MPM_OK) return st;      // the load resets the error bits
    return load_impl(h, &n, x, v, F, C, &particle_volume, on_device);
}

mpm_status mpm_load_batch(mpm_handle *h, const int64_t *counts, const float *x, const float *v, const float *F,
                          const float *C, const float *particle_volumes, int on_device) {
    mpm_status st = check_handle(h);
    if (st != MPM_OK) return st;
    if (!counts || !particle_volumes) return fail(MPM_ERR_ARG, "NULL counts or particle volumes");
    if ((st = settle_tape(h)) != MPM_OK) return st;
    return load_impl(h, counts, x, v, F, C, particle_volumes, on_device);
}

mpm_status mpm_set_env_material(mpm_handle *h, int32_t env, float E, float nu, float rho) {
    if (!h) return fail(MPM_ERR_ARG, "NULL handle");
    if (env < 0 || env >= h->n_envs) return fail(MPM_ERR_ARG, "environment %d out of range", env);
    if (!(E >= 0.f) || !(nu >= 0.f) || !(nu < 0.5f) || !(rho > 0.f))
        return fail(MPM_ERR_ARG, "need E >= 0, 0 <= nu < 0.5, rho > 0");
    h->env_E[env] = E;
    h->env_nu[env] = nu;
    h->env_rho[env] = rho;
    h->envp_dirty = true;   // applies from the next stress evaluation
    return MPM_OK;
}

mpm_status mpm_set_env_tool_pose(mpm_handle *h, int32_t env, int32_t tool_id, const double pose[6],
                                 const float shape[8]) {
    if (!h) return fail(MPM_ERR_ARG, "NULL handle");
    return set_tool_impl(h, env, tool_id, pose, shape);
}

mpm_status mpm_set_tool_pose(mpm_handle *h, int32_t tool_id, const double pose[6], const float shape[8]) {
    if (!h) return fail(MPM_ERR_ARG, "NULL handle");
    return set_tool_impl(h, 0, tool_id, pose, shape);
}

mpm_status mpm_add_sampled_field(mpm_handle *h, int32_t res, const double origin[3], double spacing,
                                 const float *samples, int on_device, int32_t *field_id) {
    mpm_status st = check_handle(h);
    if (st != MPM_OK) return st;
    if (!origin || !samples || !field_id) return fail(MPM_ERR_ARG, "NULL origin, samples or field_id");
    if (res < 1 || res > MPM_MAX_FIELD_RES) return fail(MPM_ERR_ARG, "res = %d outside [1, %d]", res, MPM_MAX_FIELD_RES);
    if (!(spacing > 0.0) || !std::isfinite(spacing)) return fail(MPM_ERR_ARG, "spacing must be finite and > 0");
    for (int a = 0; a < 3; ++a)
        if (!std::isfinite(origin[a])) return fail(MPM_ERR_ARG, "non-finite origin");
    if (h->fields.size() >= (size_t)MPM_MAX_FIELDS) return fail(MPM_ERR_CAPACITY, "at most %d sampled fields", MPM_MAX_FIELDS);
    const size_t count = (size_t)res * res * res;
    if (!on_device)
        for (size_t i = 0; i < count; ++i)
            if (std::isnan(samples[i])) return fail(MPM_ERR_ARG, "sample %zu is NaN", i);
    float *d = nullptr;
    if ((st = dalloc_t(h, &d, count)) != MPM_OK) return st;
    CK(cudaMemcpyAsync(d, samples, count * sizeof(float), on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                       h->stream));
    CK(cudaStreamSynchronize(h->stream));
    HostField f;
    f.d = d;
    f.res = res;
    for (int a = 0; a < 3; ++a) f.origin[a] = origin[a];
    f.h = spacing;
    h->fields.push_back(f);
    *field_id = (int32_t)(h->fields.size() - 1);
    return MPM_OK;
}

mpm_status mpm_step(mpm_handle *h, int32_t n_substeps) {
    mpm_status st = check_handle(h);
    if (st != MPM_OK) return st;
    if (n_substeps < 0) return fail(MPM_ERR_ARG, "n_substeps must be >= 0");
    if (!h->loaded) return fail(MPM_ERR_STATE, "no particles loaded");
    if ((st = poll_error(h, false)) != MPM_OK) return st;
    if (n_substeps == 0) return MPM_OK;
    if (h->n == 0) {
        for (auto &t : h->tools) std::memcpy(t.cur, t.tgt, sizeof t.cur);
        return MPM_OK;
    }
    for (int first = 0; first < n_substeps; first += h->sub_chunk) {
        const int m = std::min(h->sub_chunk, n_substeps - first);
        if ((st = upload_frames(h, first, m, n_substeps)) != MPM_OK) return st;
        const bool last = first + m == n_substeps;
        adapt_config(h);
        if ((st = run_chunk(h, m, last)) != MPM_OK) return st;
        if (is_fused(h)) h->step += (uint32_t)m;
    }
    h->taken += n_substeps;
    for (auto &t : h->tools) std::memcpy(t.cur, t.tgt, sizeof t.cur);
    if (!is_fused(h)) return enqueue_error_copy(h);
    CK(cudaEventRecord(h->ev_err, h->stream));     // the last launch left the error bits in h_err
    h->err_pending = true;
    return MPM_OK;
}

mpm_status mpm_synchronize(mpm_handle *h) {
    mpm_status st = check_handle(h);
    if (st != MPM_OK) return st;
    CK(cudaStreamSynchronize(h->stream));
    uint32_t err = 0;
    CK(cudaMemcpy(&err, &h->fb.ctrl->err, sizeof err, cudaMemcpyDeviceToHost));
    return status_of(err);
}

mpm_status mpm_clear_error(mpm_handle *h) {
    mpm_status st = check_handle(h);
    if (st != MPM_OK) return st;
    if ((st = settle_tape(h)) != MPM_OK) return st;
    CK(cudaMemcpyAsync(h->h_total, &h->fb.ctrl->err, sizeof(uint32_t), cudaMemcpyDeviceToHost, h->stream));
    CK(cudaMemsetAsync(&h->fb.ctrl->err, 0, sizeof(uint32_t), h->stream));
    CK(cudaStreamSynchronize(h->stream));
    // a launch whose CTAs lost one another left its counters anywhere: load again
    if (*h->h_total & kErrStall) h->loaded = false;
    *h->h_err = 0;
    h->err_pending = false;
    return MPM_OK;
}

mpm_status mpm_num_particles(mpm_handle *h, int64_t *n) {
    if (!h || !n) return fail(MPM_ERR_ARG, "NULL argument");
    *n = h->n;
    return MPM_OK;
}

mpm_status mpm_substeps_taken(mpm_handle *h, int64_t *count) {
    if (!h || !count) return fail(MPM_ERR_ARG, "NULL argument");
    *count = h->taken;
    return MPM_OK;
}

mpm_status mpm_read_particles(mpm_handle *h, float *x, float *v, float *F, float *C, int on_device) {
    mpm_status st = check_handle(h);
    if (st != MPM_OK) return st;
    if (!h->loaded) return fail(MPM_ERR_STATE, "no particles loaded");
    const size_t N = (size_t)h->n;
    if (N > 0) {
        if (on_device) {
            launch_read_out(cur_state(h), h->fb.vc, (uint32_t)N, x, v, F, C, h->elem_grid, h->stream);
        } else {
            float *sx = h->staging, *sv = sx + 3 * N, *sF = sv + 3 * N, *sC = sF + 9 * N;
            launch_read_out(cur_state(h), h->fb.vc, (uint32_t)N, x ? sx : nullptr, v ? sv : nullptr,
                            F ? sF : nullptr, C ? sC : nullptr, h->elem_grid, h->stream);
            if (x) CK(cudaMemcpyAsync(x, sx, sizeof(float) * 3 * N, cudaMemcpyDeviceToHost, h->stream));
            if (v) CK(cudaMemcpyAsync(v, sv, sizeof(float) * 3 * N, cudaMemcpyDeviceToHost, h->stream));
            if (F) CK(cudaMemcpyAsync(F, sF, sizeof(float) * 9 * N, cudaMemcpyDeviceToHost, h->stream));
            if (C) CK(cudaMemcpyAsync(C, sC, sizeof(float) * 9 * N, cudaMemcpyDeviceToHost, h->stream));
        }
        CK(cudaGetLastError());
    }
    if (!is_fused(h) || !h->err_pending) return mpm_synchronize(h);
    // whatever sets error bits on the fused pipeline (loads, sub-steps) also sends
    // them to h_err before it records ev_err
    CK(cudaStreamSynchronize(h->stream));
    CK(cudaEventSynchronize(h->ev_err));
    return status_of(*h->h_err);
}

static mpm_status ensure_dense(mpm_handle *h) {
    if (h->dense) return MPM_OK;
    return dalloc_t(h, &h->dense, (size_t)h->P.n * h->P.n * h->P.n * h->n_envs);
}

// The grid the next sub-step starts from: fused pipelines keep it in
// G[step % 3]; the split pipeline recomputes it into G[0].
static const float4 *current_grid(mpm_handle *h) {
    if (is_fused(h)) return h->fb.G[cur_m3(h)];
    cudaMemsetAsync(h->fb.G[0], 0, sizeof(float4) * (size_t)h->P.n * h->P.n * h->P.n, h->stream);
    launch_p2g_scatter(h->P, h->fb.P[0], h->fb.vc, (uint32_t)h->n, h->fb.G[0], h->fb.ctrl, h->elem_grid, h->stream);
    return h->fb.G[0];
}

mpm_status mpm_read_grid(mpm_handle *h, float *grid, int on_device) {
    mpm_status st = check_handle(h);
    if (st != MPM_OK) return st;
    if (!grid) return fail(MPM_ERR_ARG, "NULL output");
    if (!h->loaded) return fail(MPM_ERR_STATE, "no particles loaded");
    const size_t nn = (size_t)h->P.n * h->P.n * h->P.n * h->n_envs;
    const float4 *G = current_grid(h);
    if (on_device) {
        launch_grid_to_dense(h->P.n, h->P.nb, h->n_envs, G, (float4 *)grid, h->elem_grid, h->stream);
    } else {
        if ((st = ensure_dense(h)) != MPM_OK) return st;
        launch_grid_to_dense(h->P.n, h->P.nb, h->n_envs, G, h->dense, h->elem_grid, h->stream);
        CK(cudaMemcpyAsync(grid, h->dense, sizeof(float4) * nn, cudaMemcpyDeviceToHost, h->stream));
    }
    CK(cudaGetLastError());
    return mpm_synchronize(h);
}

mpm_status mpm_grid_velocity(mpm_handle *h, float *v, int on_device) {
    mpm_status st = check_handle(h);
    if (st != MPM_OK) return st;
    if (!v) return fail(MPM_ERR_ARG, "NULL output");
    if (!h->loaded) return fail(MPM_ERR_STATE, "no particles loaded");
    const size_t nn = (size_t)h->P.n * h->P.n * h->P.n * h->n_envs;
    if ((st = upload_frames(h, 0, 1, 1)) != MPM_OK) return st;
    const float4 *G = current_grid(h);
    float *outp = v;
    if (!on_device) {
        if ((st = ensure_dense(h)) != MPM_OK) return st;
        outp = reinterpret_cast<float *>(h->dense);
    }
    launch_grid_velocity_dense(h->P, G, h->d_frames, outp, h->elem_grid, h->stream);
    CK(cudaGetLastError());
    if (!on_device) CK(cudaMemcpyAsync(v, outp, sizeof(float) * 3 * nn, cudaMemcpyDeviceToHost, h->stream));
    return mpm_synchronize(h);
}

mpm_status mpm_read_order(mpm_handle *h, uint32_t *ids, uint32_t *keys) {
    mpm_status st = check_handle(h);
    if (st != MPM_OK) return st;
    if (!is_fused(h)) return fail(MPM_ERR_STATE, "the split pipeline keeps particles unsorted");
    if (!h->loaded) return fail(MPM_ERR_STATE, "no particles loaded");
    if (h->n > 0 && (!ids || !keys)) return fail(MPM_ERR_ARG, "NULL output");
    CK(cudaStreamSynchronize(h->stream));
    const int par = cur_par(h);
    const uint32_t nb = (uint32_t)h->P.nb;
    std::vector<BlockTab> tabs(h->nblocks);
    std::vector<Chunk> chunks(h->chunk_cap);
    std::vector<float4> xi((size_t)h->n);
    CK(cudaMemcpy(tabs.data(), h->fb.tabs[par], sizeof(BlockTab) * h->nblocks, cudaMemcpyDeviceToHost));
    CK(cudaMemcpy(chunks.data(), h->fb.chunks[par], sizeof(Chunk) * h->chunk_cap, cudaMemcpyDeviceToHost));
    if (h->n > 0) CK(cudaMemcpy(xi.data(), h->fb.P[par].xi, sizeof(float4) * h->n, cudaMemcpyDeviceToHost));
    size_t w = 0;
    for (uint32_t b = 0; b < h->nblocks; ++b) {
        const uint32_t e0 = (b / h->nbe) * h->nbe, bl = b % h->nbe;
        const int bx = bl % nb, by = (bl / nb) % nb, bz = bl / (nb * nb);
        for (int d = 26; d >= 0; --d) {
            const int sx = bx - (d % 3 - 1), sy = by - ((d / 3) % 3 - 1), sz = bz - (d / 9 - 1);
            if (sx < 0 || sy < 0 || sz < 0 || sx >= (int)nb || sy >= (int)nb || sz >= (int)nb) continue;
            const BlockTab &t = tabs[e0 + block_id(sx, sy, sz, nb)];
            if (t.stamp != h->step) continue;
            for (uint32_t p = 0; p < t.npass; ++p) {
                if (t.first + p >= h->chunk_cap) return fail(MPM_ERR_STATE, "corrupt run table");
                const uint2 r = chunks[t.first + p].run[d];
                for (uint32_t q = 0; q < r.y; ++q) {
                    if (w >= (size_t)h->n || r.x + q >= (size_t)h->n) return fail(MPM_ERR_STATE, "corrupt run table");
                    uint32_t id;
                    std::memcpy(&id, &xi[r.x + q].w, sizeof id);
                    ids[w] = id;
                    keys[w] = b;
                    ++w;
                }
            }
        }
    }
    if (w != (size_t)h->n) return fail(MPM_ERR_STATE, "run tables list %zu of %lld particles", w, (long long)h->n);
    return mpm_synchronize(h);
}

}  // extern "C"

// ================================================== differentiable rollout

namespace {

void image_views(float *base, int64_t n, PState &S, VCState &V) {
    const size_t n4 = 4 * (size_t)n;
    S.xi = reinterpret_cast<float4 *>(base);
    S.f0 = reinterpret_cast<float4 *>(base + n4);
    S.f1 = reinterpret_cast<float4 *>(base + 2 * n4);
    V.vc0 = reinterpret_cast<float4 *>(base + 3 * n4);
    V.vc1 = reinterpret_cast<float4 *>(base + 4 * n4);
    V.vc2 = reinterpret_cast<float4 *>(base + 5 * n4);
    S.f2 = base + 6 * n4;
}

mpm_status live_to_image(mpm_handle *h, float *img) {
    PState S;
    VCState V;
    image_views(img, h->n, S, V);
    const size_t n = (size_t)h->n;
    const PState &L = h->fb.P[0];
    CK(cudaMemcpyAsync(S.xi, L.xi, 16 * n, cudaMemcpyDeviceToDevice, h->stream));
    CK(cudaMemcpyAsync(S.f0, L.f0, 16 * n, cudaMemcpyDeviceToDevice, h->stream));
    CK(cudaMemcpyAsync(S.f1, L.f1, 16 * n, cudaMemcpyDeviceToDevice, h->stream));
    CK(cudaMemcpyAsync(S.f2, L.f2, 4 * n, cudaMemcpyDeviceToDevice, h->stream));
    CK(cudaMemcpyAsync(V.vc0, h->fb.vc.vc0, 16 * n, cudaMemcpyDeviceToDevice, h->stream));
    CK(cudaMemcpyAsync(V.vc1, h->fb.vc.vc1, 16 * n, cudaMemcpyDeviceToDevice, h->stream));
    CK(cudaMemcpyAsync(V.vc2, h->fb.vc.vc2, 16 * n, cudaMemcpyDeviceToDevice, h->stream));
    return MPM_OK;
}

// One split-pipeline sub-step of state (S, V) with grid G (P2G, grid
// operation, G2P); Gsave, if given, receives the grid the grid operation read.
mpm_status split_substep(mpm_handle *h, const PState &S, const VCState &V, float4 *G, float4 *Gsave,
                         const ToolFrame *frames) {
    const size_t nn = (size_t)h->P.n * h->P.n * h->P.n;
    const uint32_t n = (uint32_t)h->n;
    CK(cudaMemsetAsync(G, 0, sizeof(float4) * nn, h->stream));
    launch_p2g_scatter(h->P, S, V, n, G, h->fb.ctrl, h->elem_grid, h->stream);
    if (Gsave) CK(cudaMemcpyAsync(Gsave, G, sizeof(float4) * nn, cudaMemcpyDeviceToDevice, h->stream));
    launch_grid_update_dense(h->P, G, frames, h->elem_grid, h->stream);
    launch_g2p_split(h->P, S, V, n, G, h->fb.ctrl, h->elem_grid, h->stream);
    return MPM_OK;
}

template <typename T>
mpm_status ensure(mpm_handle *h, T **buf, size_t *cap, size_t count) {
    if (*cap >= count && *buf) return MPM_OK;
    mpm_status st = dalloc_t(h, buf, count);   // a smaller earlier buffer stays with the handle until destroy
    if (st == MPM_OK) *cap = count;
    return st;
}

mpm_status copy_in(float *dst, const float *src, size_t count, int on_device, cudaStream_t st) {
    if (!src) {
        CK(cudaMemsetAsync(dst, 0, sizeof(float) * count, st));
        return MPM_OK;
    }
    CK(cudaMemcpyAsync(dst, src, sizeof(float) * count, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                       st));
    return MPM_OK;
}

// CTAs of a recorded rollout's sub-steps (its forward pass and the segment replays
// of its reverse pass).
int record_grid(mpm_handle *h) {
    if (h->rec_grid == 0) h->rec_grid = h->num_sms * std::max(fused_rollout_occupancy(), 1);
    return h->rec_grid;
}

// Floats of one recorded sub-step's particles (xi, f0, f1, vc0, vc1, vc2 as
// float4; f2; the input positions, one word each), each part 16-byte aligned
size_t rs_floats(int64_t n) { return 24 * (size_t)n + 2 * (((size_t)n + 3) & ~size_t(3)); }
// Words of one recorded sub-step's block table: ranges (2 per block), the
// work list (1 per block) and the list length (padded to 4 words)
size_t rs_words(const mpm_handle *h) { return 3 * (size_t)h->nblocks + 4; }

// Whether the record of a whole rollout of nck segments of ck sub-steps is kept:
// up to 8 GiB, and a sixteenth of what the device has free beside the handle's present
// record buffers (which a larger record replaces), unless they have the room.  The
// replays that it spares cost about as much as the forward pass and share the SMs
// with the reverse sub-steps (30K particles, 100 sub-steps, gradients: 4.95 -> 4.41 ms,
// a segment recorded in one launch).
bool keeps_record(const mpm_handle *h, int64_t n, int ck, int nck) {
    const Tape &tp = h->tape;
    const size_t nn = (size_t)h->P.n * h->P.n * h->P.n, steps = (size_t)ck * nck;
    const size_t floats = rs_floats(n) * steps, grids = 2 * nn * steps, words = rs_words(h) * steps;
    if (tp.cap_rs >= floats && tp.cap_rsg >= grids && tp.cap_rsb >= words) return true;
    auto total = [](size_t f, size_t g, size_t w) { return sizeof(float) * f + sizeof(float4) * g + sizeof(uint32_t) * w; };
    const size_t bytes = total(floats, grids, words);
    size_t free_b = 0, total_b = 0;
    if (bytes > (size_t)8 << 30 || cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) return false;
    return bytes <= (free_b + total(tp.cap_rs, tp.cap_rsg, tp.cap_rsb)) / 16;
}

// Record buffers for `steps` sub-steps of n particles.  One that is too small is given
// back first, so that a handle whose rollouts grow holds the last record only; if the
// device or the caller's allocator refuses one, all are.
mpm_status reserve_record(mpm_handle *h, int64_t n, size_t steps) {
    Tape &tp = h->tape;
    const size_t nn = (size_t)h->P.n * h->P.n * h->P.n;
    const size_t floats = rs_floats(n) * steps, grids = 2 * nn * steps, words = rs_words(h) * steps;
    const bool grow_rs = tp.cap_rs < floats, grow_grid = tp.cap_rsg < grids, grow_blk = tp.cap_rsb < words;
    if (!grow_rs && !grow_grid && !grow_blk) return MPM_OK;
    CK(cudaStreamSynchronize(h->stream));
    if (h->rp_stream) CK(cudaStreamSynchronize(h->rp_stream));
    if (grow_rs) dfree(h, &tp.rs, &tp.cap_rs);
    if (grow_grid) dfree(h, &tp.rs_grid, &tp.cap_rsg);
    if (grow_blk) dfree(h, &tp.rs_blk, &tp.cap_rsb);
    mpm_status st = ensure(h, &tp.rs, &tp.cap_rs, floats);
    if (st == MPM_OK) st = ensure(h, &tp.rs_grid, &tp.cap_rsg, grids);
    if (st == MPM_OK) st = ensure(h, &tp.rs_blk, &tp.cap_rsb, words);
    if (st != MPM_OK) {
        dfree(h, &tp.rs, &tp.cap_rs);
        dfree(h, &tp.rs_grid, &tp.cap_rsg);
        dfree(h, &tp.rs_blk, &tp.cap_rsb);
        return st;
    }
    // recorded sub-steps write the grid (before and after the grid operation) over
    // their blocks' regions only; the reverse grid operation also reads the rest of the
    // blocks it lists, where it needs finite values (its adjoint there is zero)
    if (grow_grid) CK(cudaMemsetAsync(tp.rs_grid, 0, sizeof(float4) * grids, h->stream));
    return MPM_OK;
}

// Sub-step j of record buffer buf (segment sg is recorded in buffer sg % nbuf).
StepRecord step_record(mpm_handle *h, int j, int buf) {
    Tape &tp = h->tape;
    const size_t n = (size_t)tp.n;
    const size_t slot = (size_t)buf * tp.ck + j;
    float *base = tp.rs + slot * rs_floats(tp.n);
    uint32_t *w = tp.rs_blk + slot * rs_words(h);
    StepRecord r;
    r.xi = reinterpret_cast<float4 *>(base);
    r.f0 = reinterpret_cast<float4 *>(base + 4 * n);
    r.f1 = reinterpret_cast<float4 *>(base + 8 * n);
    r.vc.vc0 = reinterpret_cast<float4 *>(base + 12 * n);
    r.vc.vc1 = reinterpret_cast<float4 *>(base + 16 * n);
    r.vc.vc2 = reinterpret_cast<float4 *>(base + 20 * n);
    r.f2 = base + 24 * n;
    r.src = reinterpret_cast<uint32_t *>(base + 24 * n + ((n + 3) & ~size_t(3)));
    r.blk = reinterpret_cast<uint2 *>(w);
    r.act = w + 2 * (size_t)h->nblocks;
    r.nact = w + 3 * (size_t)h->nblocks;
    const size_t nn = (size_t)h->P.n * h->P.n * h->P.n;
    r.grid = tp.rs_grid + 2 * slot * nn;
    r.vgrid = r.grid + nn;
    r.floats = rs_floats(tp.n);
    r.words = rs_words(h);
    r.nodes = 2 * nn;
    return r;
}

// The fused state as an image by particle id: x (3n), v (3n), F (9n), C (9n); vc:
// its v and C, by position.
void id_image(mpm_handle *h, const VCState &vc, float *img) {
    const size_t n = (size_t)h->n;
    launch_read_out(cur_state(h), vc, (uint32_t)n, img, img + 3 * n, img + 6 * n, img + 15 * n, h->elem_grid,
                    h->stream);
}

mpm_status load_impl(mpm_handle *h, const int64_t *counts, const float *x, const float *v, const float *F,
                     const float *C, const float *volumes, int on_device);

// Replace the fused state by an image made with id_image.
mpm_status load_image(mpm_handle *h, const float *img) {
    const size_t n = (size_t)h->n;
    const int64_t cnt = h->n;
    const float vol = h->particle_volume;
    const int64_t taken = h->taken;
    mpm_status st = load_impl(h, &cnt, img, img + 3 * n, img + 6 * n, img + 15 * n, &vol, 1);
    h->taken = taken;
    return st;
}

// The replay stream and its events, created on first use.
mpm_status ensure_replay_stream(mpm_handle *h) {
    if (h->rp_stream) return MPM_OK;
    CK(cudaStreamCreateWithFlags(&h->rp_stream, cudaStreamNonBlocking));
    for (int b = 0; b < 2; ++b) {
        CK(cudaEventCreateWithFlags(&h->rp_rec[b], cudaEventDisableTiming));
        CK(cudaEventCreateWithFlags(&h->rp_free[b], cudaEventDisableTiming));
    }
    CK(cudaEventCreateWithFlags(&h->rp_go, cudaEventDisableTiming));
    return MPM_OK;
}

// Replay segment sg from its checkpoint with recording sub-steps, into record
// buffer sg % nbuf, on stream r (the load path runs there too).
mpm_status replay_segment(mpm_handle *h, int sg, cudaStream_t r) {
    Tape &tp = h->tape;
    const int c0 = sg * tp.ck, len = std::min(tp.ck, tp.nsub - c0), b = sg % tp.nbuf;
    cudaStream_t keep = h->stream;
    h->stream = r;
    mpm_status st = load_image(h, tp.ckpt + (size_t)sg * tp.image);
    if (st == MPM_OK) {
        for (int j = 0; j < len; ++j) {
            launch_fused_step_record(h->P, h->fb, tp.frames + (size_t)(c0 + j) * tp.ntools, step_record(h, j, b),
                                     1, record_grid(h), r);
            h->step += 1u;
        }
    }
    h->stream = keep;
    return st;
}

// Reverse pass of a rollout recorded on the fused pipeline.  Segment by
// segment, last first: reverse the segment's sub-steps from its record with
// the block-sorted reverse sub-step (G2P of sub-step k and P2G of sub-step
// k+1) and the reverse grid operation of sub-step k; finally the reverse of
// the first sub-step's P2G.  The record of a segment is made by replaying it
// from its checkpoint; with two record buffers the replays run on their own
// stream one segment ahead, beside the reverse of the segment after.  The
// last segment's record comes from the forward pass.  Replays leave their own
// state in place of the live one.
mpm_status fused_reverse(mpm_handle *h, const AdjState &A, int nck) {
    Tape &tp = h->tape;
    const int nt = tp.ntools;
    const size_t n = (size_t)tp.n;
    const size_t nn = (size_t)h->P.n * h->P.n * h->P.n;
    const size_t nbk = h->nblocks;
    cudaStream_t s = h->stream;
    if (h->rev_grid == 0) h->rev_grid = h->num_sms * std::max(reverse_step_ctas_per_sm(), 1);
    float4 *gnext = tp.gbar, *gcur = tp.gb2;     // dL/d(m, mv) of G_{k+1}; dL/dV_k, then dL/d(m, mv) of G_k
    // both start clean; afterwards only the blocks a sub-step touched are cleared.
    // The touched-block list of sub-step k lives in slot k % 3 (8 entries per
    // work-list block, then the three slots' work-list lengths); the reverse grid
    // operation of sub-step k clears the blocks of sub-step k+1.
    CK(cudaMemsetAsync(gnext, 0, sizeof(float4) * nn, s));
    CK(cudaMemsetAsync(gcur, 0, sizeof(float4) * nn, s));
    uint32_t *stamp = tp.touch, *lists = tp.touch + nbk, *counts = lists + 24 * nbk;
    CK(cudaMemsetAsync(counts, 0, 3 * sizeof(uint32_t), s));
    mpm_status st;
    if ((st = ensure(h, &tp.lame_part, &tp.cap_lame, 2 * (size_t)h->rev_grid)) != MPM_OK) return st;
    CK(cudaMemsetAsync(tp.lame_part, 0, sizeof(double) * 2 * h->rev_grid, s));
    // the state adjoints between the sub-steps of a segment, by position (two
    // buffers of 3 n float4: the incoming one and the outgoing one)
    if ((st = ensure(h, &tp.lp, &tp.cap_lp, 6 * n)) != MPM_OK) return st;
    float4 *lp_in = tp.lp, *lp_out = tp.lp + 3 * n;
    // the reverse grid operation: one wave of 3 CTAs per SM (a node per thread
    // over 8 list entries per work-list block, most of them empty)
    const int adj_grid_ctas = 3 * h->num_sms;
    const bool have_all = tp.nbuf == nck;     // every segment's record comes from the forward pass
    const bool have_last = tp.last_recorded;
    tp.last_recorded = false;     // replays overwrite the record buffers
    const bool ahead = tp.nbuf == 2 && !have_all;
    cudaStream_t r = s;
    if (ahead) {
        if ((st = ensure_replay_stream(h)) != MPM_OK) return st;
        r = h->rp_stream;
        CK(cudaEventRecord(h->rp_go, s));       // replays follow everything issued so far
        CK(cudaStreamWaitEvent(r, h->rp_go, 0));
        // the first segments: the last one (unless the forward pass recorded it)
        // and the one before it, into the two buffers
        for (int sg = nck - 1; sg >= std::max(nck - 2, 0); --sg) {
            if (sg == nck - 1 && have_last) continue;
            if ((st = replay_segment(h, sg, r)) != MPM_OK) return st;
            CK(cudaEventRecord(h->rp_rec[sg % 2], r));
        }
    }
    for (int sg = nck - 1; sg >= 0; --sg) {
        const int c0 = sg * tp.ck, len = std::min(tp.ck, tp.nsub - c0), b = sg % tp.nbuf;
        const bool replayed = !have_all && !(sg == nck - 1 && have_last);
        if (replayed) {
            if (ahead) {
                CK(cudaStreamWaitEvent(s, h->rp_rec[b], 0));
            } else if ((st = replay_segment(h, sg, s)) != MPM_OK) {
                return st;
            }
        }
        for (int j = len - 1; j >= 0; --j) {
            const int k = c0 + j;
            const int sk = k % 3, sk1 = (k + 1) % 3;
            ReverseArgs R{};
            R.rec = step_record(h, j, b);
            R.gbar_next = gnext;
            R.vbar = gcur;
            R.lam = A;
            R.lp_in = lp_in;
            R.lp_out = lp_out;
            R.np = (uint32_t)n;
            R.lam_in_by_id = j == len - 1;
            R.lam_out_by_id = j == 0;
            R.lame_part = tp.lame_part;
            R.stamp = stamp;
            R.sv = ++tp.touch_sv;
            R.touch_list = lists + (size_t)sk * 8 * nbk;
            R.touch_n = counts + sk;
            // a segment's first reverse launch follows its replay (and the wait for it)
            // in full; the others are programmatic dependents of the launch before
            launch_reverse_step(k + 1 < tp.nsub, true, h->P, R, h->rev_grid, s, j < len - 1);
            AdjGridLists L;
            L.list = R.touch_list;
            L.nlist = R.touch_n;
            L.zlist = lists + (size_t)sk1 * 8 * nbk;
            L.znlist = counts + sk1;
            L.zbuf = gnext;
            if (j > 0) {
                L.prefetch = step_record(h, j - 1, b).xi;     // sub-step k-1's particles, one slab
                L.prefetch_bytes = sizeof(float) * rs_floats(tp.n);
            }
            launch_adj_grid(h->P, R.rec.grid, tp.frames + (size_t)k * nt, gcur, tp.red + 2 + (size_t)k * nt * 18,
                            adj_grid_ctas, s, L);
            std::swap(gnext, gcur);
            std::swap(lp_in, lp_out);
        }
        if (ahead && sg >= 2) {
            // buffer b is free once this segment's reverse is done: replay sg - 2 into it
            CK(cudaEventRecord(h->rp_free[b], s));
            CK(cudaStreamWaitEvent(r, h->rp_free[b], 0));
            if ((st = replay_segment(h, sg - 2, r)) != MPM_OK) return st;
            CK(cudaEventRecord(h->rp_rec[b], r));
        }
    }
    // the first sub-step's P2G at the initial state (its v and C from checkpoint 0)
    ReverseArgs R{};
    R.rec = step_record(h, 0, 0);
    R.gbar_next = gnext;
    R.lam = A;
    R.v0 = tp.ckpt + 3 * n;
    R.C0 = tp.ckpt + 15 * n;
    R.np = (uint32_t)n;
    R.lam_in_by_id = 1;
    R.lam_out_by_id = 1;
    R.lame_part = tp.lame_part;
    launch_reverse_step(true, false, h->P, R, h->rev_grid, s, true);
    CK(cudaGetLastError());
    return MPM_OK;
}

mpm_status copy_out(float *dst, const float *src, size_t count, int on_device, cudaStream_t st) {
    if (!dst) return MPM_OK;
    CK(cudaMemcpyAsync(dst, src, sizeof(float) * count, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                       st));
    return MPM_OK;
}

}  // namespace

extern "C" {

mpm_status mpm_tape_record(mpm_handle *h, int32_t n_substeps, const double *poses, int32_t checkpoint_every) {
    mpm_status st = check_handle(h);
    if (st != MPM_OK) return st;
    if (h->n_envs != 1) return fail(MPM_ERR_STATE, "mpm_tape_record needs a handle with one environment");
    if (!h->loaded) return fail(MPM_ERR_STATE, "no particles loaded");
    if (n_substeps < 1) return fail(MPM_ERR_ARG, "n_substeps must be >= 1");
    if (checkpoint_every < 1) return fail(MPM_ERR_ARG, "checkpoint_every must be >= 1");
    const int nt = tool_stride(h);
    if (nt > 0 && !poses) return fail(MPM_ERR_ARG, "NULL poses");
    for (size_t i = 0; i < (size_t)n_substeps * nt * 6; ++i)
        if (!std::isfinite(poses[i])) return fail(MPM_ERR_ARG, "non-finite pose");
    if ((st = poll_error(h, false)) != MPM_OK) return st;
    Tape &tp = h->tape;
    tp.valid = false;
    tp.last_recorded = false;
    const int64_t n = h->n;
    const int ck = std::min(checkpoint_every, n_substeps);
    const int nck = (n_substeps + ck - 1) / ck;
    const size_t nn = (size_t)h->P.n * h->P.n * h->P.n;
    tp.fused = is_fused(h);
    if (tp.fused) {
        tp.image = 24 * (size_t)n;
        if ((st = ensure(h, &tp.ckpt, &tp.cap_ckpt, tp.image * nck)) != MPM_OK) return st;
        if ((st = ensure(h, &tp.final_img, &tp.cap_final, tp.image)) != MPM_OK) return st;
        // a record buffer for every segment where that is little memory; otherwise two
        // when there are several: the reverse pass replays a segment into one while
        // it reverses the one in the other
        int nbuf = keeps_record(h, n, ck, nck) ? nck : std::min(nck, 2);
        st = reserve_record(h, n, (size_t)ck * nbuf);
        if (st == MPM_ERR_ALLOC && nbuf > 2) {
            cudaGetLastError();
            nbuf = 2;
            st = reserve_record(h, n, (size_t)ck * nbuf);
        }
        if (st != MPM_OK) return st;
        tp.nbuf = nbuf;
        if ((st = ensure(h, &tp.gbar, &tp.cap_gb, nn)) != MPM_OK) return st;
        size_t one = tp.cap_gb;
        if ((st = ensure(h, &tp.gb2, &one, nn)) != MPM_OK) return st;
        const size_t tw = 25 * (size_t)h->nblocks + 3;
        if (tp.cap_touch < tw) {
            if ((st = ensure(h, &tp.touch, &tp.cap_touch, tw)) != MPM_OK) return st;
            CK(cudaMemsetAsync(tp.touch, 0, sizeof(uint32_t) * tw, h->stream));
            tp.touch_sv = 0;
        }
    } else {
        tp.image = 24 * (size_t)n + (((size_t)n + 3) & ~size_t(3));
        if ((st = ensure(h, &tp.ckpt, &tp.cap_ckpt, tp.image * nck)) != MPM_OK) return st;
        if ((st = ensure(h, &tp.seg, &tp.cap_seg, tp.image * ck)) != MPM_OK) return st;
        if ((st = ensure(h, &tp.seg_grid, &tp.cap_grid, nn * ck)) != MPM_OK) return st;
        if ((st = ensure(h, &tp.seg_vel, &tp.cap_vel, nn * ck)) != MPM_OK) return st;
        size_t one = nn;
        if ((st = ensure(h, &tp.gv, &one, nn)) != MPM_OK) return st;
        one = nn;
        if ((st = ensure(h, &tp.gbar, &one, nn)) != MPM_OK) return st;
    }
    if ((st = ensure(h, &tp.abar, &tp.cap_abar, 24 * (size_t)n)) != MPM_OK) return st;
    if ((st = ensure(h, &tp.frames, &tp.cap_frames, (size_t)n_substeps * std::max(nt, 1))) != MPM_OK) return st;
    if ((st = ensure(h, &tp.red, &tp.cap_red, 2 + (size_t)n_substeps * nt * 18)) != MPM_OK) return st;
    if ((st = upload_env_params(h)) != MPM_OK) return st;
    // frames: one sub-step per pose, from each tool's current pose
    tp.pose_init.assign((size_t)nt * 6, 0.0);
    tp.poses.assign(poses, poses + (size_t)n_substeps * nt * 6);
    for (int t = 0; t < nt; ++t) std::memcpy(&tp.pose_init[6 * t], h->tools[t].cur, 6 * sizeof(double));
    std::vector<ToolFrame> hf((size_t)n_substeps * std::max(nt, 1));
    for (int k = 0; k < n_substeps && nt > 0; ++k) {
        for (int t = 0; t < nt; ++t) std::memcpy(h->tools[t].tgt, poses + ((size_t)k * nt + t) * 6, 6 * sizeof(double));
        fill_frames(h, 0, 1, 1, nt, &hf[(size_t)k * nt]);
        for (int t = 0; t < nt; ++t) std::memcpy(h->tools[t].cur, h->tools[t].tgt, 6 * sizeof(double));
    }
    if (nt > 0) CK(cudaMemcpy(tp.frames, hf.data(), sizeof(ToolFrame) * hf.size(), cudaMemcpyHostToDevice));
    tp.E = h->env_E[0];
    tp.nu = h->env_nu[0];
    tp.mat = h->envp_host[0];
    if (tp.fused) {
        // checkpoints by particle id; v and C of a checkpointed state are written by
        // the sub-step before it.  The last segment runs with recording sub-steps,
        // so that the reverse pass starts without replaying it (step_record lays
        // the records out for tp.n particles and tp.ck sub-steps per buffer).
        tp.n = n;
        tp.ck = ck;
        const int c_last = (nck - 1) * ck, b_last = (nck - 1) % tp.nbuf;
        const bool all = tp.nbuf == nck;
        for (int k = 0; k < n_substeps;) {
            // a recording sub-step leaves v and C in its record
            const bool recorded = k > 0 && (all || k > c_last);
            const VCState before = recorded ? step_record(h, (k - 1) % ck, (k - 1) / ck % tp.nbuf).vc : h->fb.vc;
            if (k % ck == 0) id_image(h, before, tp.ckpt + (size_t)(k / ck) * tp.image);
            int m = 1;
            if (all || k >= c_last) {
                m = std::min(ck, n_substeps - k);
                launch_fused_step_record(h->P, h->fb, tp.frames + (size_t)k * nt, step_record(h, 0, k / ck % tp.nbuf),
                                         m, record_grid(h), h->stream);
            } else {
                m = std::min(ck, n_substeps - k);
                launch_fused_steps_rollout(h->P, h->fb, tp.frames + (size_t)k * nt, m, record_grid(h), h->stream);
            }
            h->step += (uint32_t)m;
            k += m;
        }
        // the last sub-step kept v and C in its record, by output position: they
        // become the live state's
        const VCState rv = step_record(h, n_substeps - 1 - c_last, b_last).vc;
        CK(cudaMemcpyAsync(h->fb.vc.vc0, rv.vc0, 16 * (size_t)n, cudaMemcpyDeviceToDevice, h->stream));
        CK(cudaMemcpyAsync(h->fb.vc.vc1, rv.vc1, 16 * (size_t)n, cudaMemcpyDeviceToDevice, h->stream));
        CK(cudaMemcpyAsync(h->fb.vc.vc2, rv.vc2, 16 * (size_t)n, cudaMemcpyDeviceToDevice, h->stream));
        id_image(h, h->fb.vc, tp.final_img);
        tp.last_recorded = true;
        tp.end_step = h->step;
    } else {
        for (int k = 0; k < n_substeps; ++k) {
            if (k % ck == 0 && (st = live_to_image(h, tp.ckpt + (size_t)(k / ck) * tp.image)) != MPM_OK) return st;
            if ((st = split_substep(h, h->fb.P[0], h->fb.vc, h->fb.G[0], nullptr, tp.frames + (size_t)k * nt)) !=
                MPM_OK)
                return st;
        }
    }
    CK(cudaGetLastError());
    h->taken += n_substeps;
    tp.nsub = n_substeps;
    tp.ck = ck;
    tp.ntools = nt;
    tp.n = n;
    tp.valid = true;
    tp.settled = !tp.fused;
    return enqueue_error_copy(h);
}

mpm_status mpm_tape_backward(mpm_handle *h, const float *x_bar, const float *v_bar, const float *F_bar,
                             const float *C_bar, int on_device, double *grad_material, double *grad_poses,
                             float *x0_bar, float *v0_bar, float *F0_bar, float *C0_bar) {
    mpm_status st = check_handle(h);
    if (st != MPM_OK) return st;
    Tape &tp = h->tape;
    if (!tp.valid || tp.n != h->n) return fail(MPM_ERR_STATE, "no recorded rollout (mpm_tape_record) for this state");
    if (tool_stride(h) != tp.ntools || h->env_E[0] != tp.E || h->env_nu[0] != tp.nu)
        return fail(MPM_ERR_STATE, "tools or material changed since mpm_tape_record");
    if ((st = settle_tape(h)) != MPM_OK) return st;
    if ((st = poll_error(h, !tp.valid)) != MPM_OK) return st;
    // The rollout is reversed, and replayed, with the material it was recorded with:
    // what the handle's table holds now may have been set or loaded since, and the
    // tool stride may be another's.
    if ((st = upload_env_params(h)) != MPM_OK) return st;
    struct Material {
        DevParams &P;
        const EnvParams *live;
        ~Material() { P.envp = live; }
    } material{h->P, h->P.envp};
    const bool same_material = std::memcmp(&tp.mat, &h->envp_host[0], sizeof tp.mat) == 0;
    if (!same_material) {
        if (!tp.d_mat && (st = dalloc_t(h, &tp.d_mat, 1)) != MPM_OK) return st;
        CK(cudaMemcpyAsync(tp.d_mat, &tp.mat, sizeof tp.mat, cudaMemcpyHostToDevice, h->stream));
        h->P.envp = tp.d_mat;
    }
    const int64_t n = tp.n;
    const int nt = tp.ntools;
    const size_t nn = (size_t)h->P.n * h->P.n * h->P.n;
    cudaStream_t s = h->stream;
    AdjState A;
    A.x = tp.abar;
    A.v = tp.abar + 3 * (size_t)n;
    A.C = tp.abar + 6 * (size_t)n;
    A.F = tp.abar + 15 * (size_t)n;
    if ((st = copy_in(A.x, x_bar, 3 * (size_t)n, on_device, s)) != MPM_OK) return st;
    if ((st = copy_in(A.v, v_bar, 3 * (size_t)n, on_device, s)) != MPM_OK) return st;
    if ((st = copy_in(A.F, F_bar, 9 * (size_t)n, on_device, s)) != MPM_OK) return st;
    if ((st = copy_in(A.C, C_bar, 9 * (size_t)n, on_device, s)) != MPM_OK) return st;
    const size_t nred = 2 + (size_t)tp.nsub * nt * 18;
    CK(cudaMemsetAsync(tp.red, 0, sizeof(double) * nred, s));
    const int nck = (tp.nsub + tp.ck - 1) / tp.ck;
    if (tp.fused) {
        const bool replayed = tp.nbuf != nck;
        if ((st = fused_reverse(h, A, nck)) != MPM_OK) return st;
        h->P.envp = material.live;
        // the live state back to the rollout's end, which it still is without replays and
        // with nothing stepped, loaded or set since
        if ((replayed || h->step != tp.end_step || !same_material) && (st = load_image(h, tp.final_img)) != MPM_OK)
            return st;
    }
    for (int sg = tp.fused ? -1 : nck - 1; sg >= 0; --sg) {
        const int c0 = sg * tp.ck, len = std::min(tp.ck, tp.nsub - c0);
        CK(cudaMemcpyAsync(tp.seg, tp.ckpt + (size_t)sg * tp.image, sizeof(float) * tp.image, cudaMemcpyDeviceToDevice,
                           s));
        // replay the segment, keeping every state, the grid each grid operation
        // read and the velocities it wrote
        for (int j = 0; j < len; ++j) {
            PState Sj;
            VCState Vj;
            image_views(tp.seg + (size_t)j * tp.image, n, Sj, Vj);
            float4 *Gj = tp.seg_grid + (size_t)j * nn, *Uj = tp.seg_vel + (size_t)j * nn;
            CK(cudaMemsetAsync(Gj, 0, sizeof(float4) * nn, s));
            launch_p2g_scatter(h->P, Sj, Vj, (uint32_t)n, Gj, h->fb.ctrl, h->elem_grid, s);
            launch_grid_update_dense_to(h->P, Gj, Uj, tp.frames + (size_t)(c0 + j) * nt, h->elem_grid, s);
            if (j + 1 < len) {
                float *next = tp.seg + (size_t)(j + 1) * tp.image;
                CK(cudaMemcpyAsync(next, tp.seg + (size_t)j * tp.image, sizeof(float) * tp.image,
                                   cudaMemcpyDeviceToDevice, s));
                PState Sn;
                VCState Vn;
                image_views(next, n, Sn, Vn);
                launch_g2p_split(h->P, Sn, Vn, (uint32_t)n, Uj, h->fb.ctrl, h->elem_grid, s);
            }
        }
        // reverse the segment's sub-steps
        for (int j = len - 1; j >= 0; --j) {
            const int k = c0 + j;
            PState Sj;
            VCState Vj;
            image_views(tp.seg + (size_t)j * tp.image, n, Sj, Vj);
            const float4 *Gj = tp.seg_grid + (size_t)j * nn, *Uj = tp.seg_vel + (size_t)j * nn;
            const ToolFrame *fr = tp.frames + (size_t)k * nt;
            // v and C after sub-step k: the next image of the segment or the next
            // checkpoint (after the last sub-step none is kept: formed again)
            VCState Vk1{};
            PState Sk1;
            if (j + 1 < len)
                image_views(tp.seg + (size_t)(j + 1) * tp.image, n, Sk1, Vk1);
            else if (sg + 1 < nck)
                image_views(tp.ckpt + (size_t)(sg + 1) * tp.image, n, Sk1, Vk1);
            CK(cudaMemsetAsync(tp.gbar, 0, sizeof(float4) * nn, s));
            launch_adj_g2p(h->P, Sj, (uint32_t)n, Uj, A, tp.gbar, Vk1, h->elem_grid, s);
            launch_adj_grid(h->P, Gj, fr, tp.gbar, tp.red + 2 + (size_t)k * nt * 18, h->elem_grid, s);
            launch_adj_p2g(h->P, Sj, Vj, (uint32_t)n, tp.gbar, A, tp.red, h->elem_grid, s);
        }
    }
    CK(cudaGetLastError());
    if ((st = copy_out(x0_bar, A.x, 3 * (size_t)n, on_device, s)) != MPM_OK) return st;
    if ((st = copy_out(v0_bar, A.v, 3 * (size_t)n, on_device, s)) != MPM_OK) return st;
    if ((st = copy_out(F0_bar, A.F, 9 * (size_t)n, on_device, s)) != MPM_OK) return st;
    if ((st = copy_out(C0_bar, A.C, 9 * (size_t)n, on_device, s)) != MPM_OK) return st;
    std::vector<double> red(nred);
    CK(cudaMemcpyAsync(red.data(), tp.red, sizeof(double) * nred, cudaMemcpyDeviceToHost, s));
    std::vector<double> lame_part(tp.fused ? 2 * (size_t)h->rev_grid : 0);
    if (tp.fused)
        CK(cudaMemcpyAsync(lame_part.data(), tp.lame_part, sizeof(double) * lame_part.size(), cudaMemcpyDeviceToHost,
                           s));
    if ((st = enqueue_error_copy(h)) != MPM_OK) return st;
    CK(cudaStreamSynchronize(s));
    if ((st = poll_error(h, true)) != MPM_OK) return st;
    for (size_t c = 0; c + 1 < lame_part.size(); c += 2) {
        red[0] += lame_part[c];
        red[1] += lame_part[c + 1];
    }
    if (grad_material) {   // Eq. 6 backwards
        const double E = tp.E, nu = tp.nu, D = (1.0 + nu) * (1.0 - 2.0 * nu);
        grad_material[0] = red[0] / (2.0 * (1.0 + nu)) + red[1] * nu / D;
        grad_material[1] = -red[0] * E / (2.0 * (1.0 + nu) * (1.0 + nu)) + red[1] * E * (1.0 + 2.0 * nu * nu) / (D * D);
    }
    if (grad_poses) {
        std::fill(grad_poses, grad_poses + (size_t)tp.nsub * nt * 6, 0.0);
        const double span = (double)h->cfg.dt;
        for (int k = 0; k < tp.nsub; ++k)
            for (int t = 0; t < nt; ++t) {
                if (h->tools[t].kind == MPM_TOOL_NONE) continue;
                const double *fb = &red[2 + ((size_t)k * nt + t) * 18];
                const double *p0 = k == 0 ? &tp.pose_init[6 * t] : &tp.poses[((size_t)(k - 1) * nt + t) * 6];
                const double *p1 = &tp.poses[((size_t)k * nt + t) * 6];
                Dual<12> a[6], b[6], R[9], T[3], u[3], w[3];
                for (int i = 0; i < 6; ++i) {
                    a[i] = Dual<12>(p0[i]);
                    a[i].d[i] = 1.0;
                    b[i] = Dual<12>(p1[i]);
                    b[i].d[6 + i] = 1.0;
                }
                call_frame(a, b, 1.0, span, R, T, u, w);
                const Dual<12> *fr[18] = {&R[0], &R[1], &R[2], &R[3], &R[4], &R[5], &R[6], &R[7], &R[8],
                                          &T[0], &T[1], &T[2], &u[0], &u[1], &u[2], &w[0], &w[1], &w[2]};
                double g[12] = {};
                for (int f = 0; f < 18; ++f)
                    for (int i = 0; i < 12; ++i) g[i] += fb[f] * fr[f]->d[i];
                if (k > 0)
                    for (int i = 0; i < 6; ++i) grad_poses[((size_t)(k - 1) * nt + t) * 6 + i] += g[i];
                for (int i = 0; i < 6; ++i) grad_poses[((size_t)k * nt + t) * 6 + i] += g[6 + i];
            }
    }
    return MPM_OK;
}

mpm_status mpm_tape_read_substep(mpm_handle *h, int32_t j, float *x, float *v, float *F, float *C, float *grid,
                                 int on_device) {
    mpm_status st = check_handle(h);
    if (st != MPM_OK) return st;
    Tape &tp = h->tape;
    if (!tp.valid || !tp.fused || !tp.last_recorded || tp.n != h->n)
        return fail(MPM_ERR_STATE, "no recorded segment (a fused-pipeline mpm_tape_record, before mpm_tape_backward)");
    const int nck = (tp.nsub + tp.ck - 1) / tp.ck, c_last = (nck - 1) * tp.ck, len = tp.nsub - c_last;
    if (j < 0 || j >= len) return fail(MPM_ERR_ARG, "j outside the last segment of the record");
    if ((st = poll_error(h, false)) != MPM_OK) return st;
    const size_t n = (size_t)tp.n;
    cudaStream_t s = h->stream;
    // host outputs are staged in the adjoint buffer, which mpm_tape_backward sets anew
    float *ox = x, *ov = v, *oF = F, *oC = C;
    if (!on_device) {
        ox = x ? tp.abar : nullptr;
        ov = v ? tp.abar + 3 * n : nullptr;
        oF = F ? tp.abar + 6 * n : nullptr;
        oC = C ? tp.abar + 15 * n : nullptr;
    }
    const int b = (nck - 1) % tp.nbuf;
    const StepRecord r = step_record(h, j, b);
    if (ox || oF) launch_read_out(PState{r.xi, r.f0, r.f1, r.f2}, r.vc, (uint32_t)n, ox, nullptr, oF, nullptr,
                                  h->elem_grid, s);
    if (ov || oC) {
        if (j > 0) {
            // v and C as the sub-step before wrote them (its record holds the ids at the same positions)
            const StepRecord q = step_record(h, j - 1, b);
            launch_read_out(PState{q.xi, q.f0, q.f1, q.f2}, q.vc, (uint32_t)n, nullptr, ov, nullptr, oC, h->elem_grid, s);
        } else {
            const float *ck = tp.ckpt + (size_t)(nck - 1) * tp.image;     // the segment's checkpoint, by id
            if (ov) CK(cudaMemcpyAsync(ov, ck + 3 * n, sizeof(float) * 3 * n, cudaMemcpyDeviceToDevice, s));
            if (oC) CK(cudaMemcpyAsync(oC, ck + 15 * n, sizeof(float) * 9 * n, cudaMemcpyDeviceToDevice, s));
        }
    }
    if (!on_device) {
        if (x) CK(cudaMemcpyAsync(x, ox, sizeof(float) * 3 * n, cudaMemcpyDeviceToHost, s));
        if (v) CK(cudaMemcpyAsync(v, ov, sizeof(float) * 3 * n, cudaMemcpyDeviceToHost, s));
        if (F) CK(cudaMemcpyAsync(F, oF, sizeof(float) * 9 * n, cudaMemcpyDeviceToHost, s));
        if (C) CK(cudaMemcpyAsync(C, oC, sizeof(float) * 9 * n, cudaMemcpyDeviceToHost, s));
    }
    if (grid) {
        const size_t nn = (size_t)h->P.n * h->P.n * h->P.n;
        if (on_device) {
            launch_grid_to_dense(h->P.n, h->P.nb, 1, r.grid, reinterpret_cast<float4 *>(grid), h->elem_grid, s);
        } else {
            if ((st = ensure_dense(h)) != MPM_OK) return st;
            launch_grid_to_dense(h->P.n, h->P.nb, 1, r.grid, h->dense, h->elem_grid, s);
            CK(cudaMemcpyAsync(grid, h->dense, sizeof(float4) * nn, cudaMemcpyDeviceToHost, s));
        }
    }
    CK(cudaGetLastError());
    return mpm_synchronize(h);
}

}  // extern "C"

// =========================================================== kernel tuning

namespace {

mpm_status apply_kernel_config(mpm_handle *h, int config) {
    const int occ = fused_step_occupancy(config);
    CK(cudaGetLastError());
    if (occ < 1) return fail(MPM_ERR_ARG, "kernel configuration %d does not fit on this device", config);
    h->kernel_config = config;
    h->fused_grid = h->num_sms * occ;
    return MPM_OK;
}

}  // namespace

extern "C" {

mpm_status mpm_set_kernel_config(mpm_handle *h, int32_t config) {
    mpm_status st = check_handle(h);
    if (st != MPM_OK) return st;
    if (config < 0 || config >= MPM_KERNEL_CONFIGS) return fail(MPM_ERR_ARG, "kernel configuration %d out of range", config);
    st = apply_kernel_config(h, config);
    if (st != MPM_OK) return st;
    h->config_set = true;
    h->few_blocks = h->by_volume = false;
    if (is_fused(h)) ensure_runs(h);      // or, refused, half of a block's capacity with 128 threads
    return MPM_OK;
}

mpm_status mpm_get_kernel_config(mpm_handle *h, int32_t *config, int32_t *threads, int32_t *ctas) {
    mpm_status st = check_handle(h);
    if (st != MPM_OK) return st;
    if (config) *config = h->config_set ? h->kernel_config : h->tuned;
    if (threads) *threads = fused_step_threads(h->kernel_config);
    if (ctas) *ctas = h->fused_grid;
    return MPM_OK;
}

// timed calls per configuration in mpm_autotune (their median is compared)
constexpr int kTuneReps = 3;

mpm_status mpm_autotune(mpm_handle *h, int32_t n_substeps, float *times_ms, int32_t *best) {
    mpm_status st = check_handle(h);
    if (st != MPM_OK) return st;
    if (!is_fused(h)) return fail(MPM_ERR_STATE, "mpm_autotune tunes the fused pipeline");
    if (!h->loaded) return fail(MPM_ERR_STATE, "no particles loaded");
    if (n_substeps < 1) return fail(MPM_ERR_ARG, "n_substeps must be >= 1");
    if ((st = poll_error(h, true)) != MPM_OK) return st;
    if (times_ms)
        for (int c = 0; c < MPM_KERNEL_CONFIGS; ++c) times_ms[c] = -1.f;
    if (h->n == 0) {
        if (best) *best = h->config_set ? h->kernel_config : h->tuned;
        return MPM_OK;
    }
    // snapshot of the state, the tools and the counters; every trial starts from it
    const size_t n = (size_t)h->n;
    if ((st = ensure(h, &h->tune_snap, &h->tune_cap, 24 * n)) != MPM_OK) return st;
    float *snap = h->tune_snap;
    float *sx = snap, *sv = snap + 3 * n, *sF = snap + 6 * n, *sC = snap + 15 * n;
    if ((st = mpm_read_particles(h, sx, sv, sF, sC, 1)) != MPM_OK) return st;
    const std::vector<HostTool> tools0 = h->tools;
    const int64_t taken0 = h->taken;
    std::vector<int64_t> counts(h->n_envs);
    std::vector<float> vols(h->n_envs);
    for (int e = 0; e < h->n_envs; ++e) {
        counts[e] = (int64_t)h->env_off[e + 1] - (int64_t)h->env_off[e];
        vols[e] = (float)h->env_vol[e];
    }
    const int start = h->kernel_config;
    const bool start_set = h->config_set;
    cudaEvent_t a = nullptr, b = nullptr;
    if (cudaEventCreate(&a) != cudaSuccess || cudaEventCreate(&b) != cudaSuccess) {
        if (a) cudaEventDestroy(a);
        return fail(MPM_ERR_CUDA, "cudaEventCreate failed");
    }
    h->config_set = true;     // the trials' loads keep the trial's configuration
    auto restore = [&]() -> mpm_status {
        h->tools = tools0;
        return load_impl(h, counts.data(), sx, sv, sF, sC, vols.data(), 1);
    };
    int pick = start, selectable = 0;
    float best_ms = 3.0e38f, selectable_ms = 3.0e38f;
    // the selectable ones, and the library's own where a load would take it
    const int last = choose_config(h) == kConfigT512 ? kConfigT512 : MPM_KERNEL_CONFIGS - 1;
    for (int c = 0; c <= last && st == MPM_OK; ++c) {
        if (fused_step_occupancy(c) < 1) continue;
        if ((st = apply_kernel_config(h, c)) != MPM_OK) break;
        if ((st = restore()) != MPM_OK) break;
        if ((st = mpm_step(h, n_substeps)) != MPM_OK) break;      // captures the graphs
        // the median of kTuneReps timed calls
        float reps[kTuneReps];
        for (int r = 0; r < kTuneReps && st == MPM_OK; ++r) {
            h->tools = tools0;
            cudaEventRecord(a, h->stream);
            if ((st = mpm_step(h, n_substeps)) != MPM_OK) break;
            cudaEventRecord(b, h->stream);
            if (cudaEventSynchronize(b) != cudaSuccess) { st = fail(MPM_ERR_CUDA, "cudaEventSynchronize failed"); break; }
            if ((st = poll_error(h, true)) != MPM_OK) break;
            reps[r] = 0.f;
            cudaEventElapsedTime(&reps[r], a, b);
        }
        if (st != MPM_OK) break;
        std::sort(reps, reps + kTuneReps);
        const float ms = reps[kTuneReps / 2];
        if (times_ms && c < MPM_KERNEL_CONFIGS) times_ms[c] = ms;
        if (ms < best_ms) { best_ms = ms; pick = c; }
        if (c < MPM_KERNEL_CONFIGS && ms < selectable_ms) { selectable_ms = ms; selectable = c; }
    }
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    mpm_status st2 = apply_kernel_config(h, st == MPM_OK ? pick : start);
    if (st != MPM_OK) h->config_set = start_set;
    else if (pick == kConfigT512) h->config_set = false;     // the load's choice again
    if (st2 == MPM_OK) st2 = restore();
    h->taken = taken0;
    if (st != MPM_OK) return st;
    if (st2 != MPM_OK) return st2;
    // what is reported can be set on another handle: also where a load's own choice won
    h->tuned = selectable;
    if (best) *best = selectable;
    return MPM_OK;
}

}  // extern "C"

// ===================================================== surface extraction

extern "C" {

mpm_status mpm_extract_surface(mpm_handle *h, int32_t env, float iso, float *tri, int64_t max_tri, int64_t *n_tri,
                               int on_device) {
    mpm_status st = check_handle(h);
    if (st != MPM_OK) return st;
    if (!n_tri) return fail(MPM_ERR_ARG, "NULL n_tri");
    if (env < 0 || env >= h->n_envs) return fail(MPM_ERR_ARG, "environment %d out of range", env);
    if (max_tri < 0 || (max_tri > 0 && !tri)) return fail(MPM_ERR_ARG, "need max_tri >= 0 and an output array");
    if (!std::isfinite(iso)) return fail(MPM_ERR_ARG, "non-finite iso");
    if (!h->loaded) return fail(MPM_ERR_STATE, "no particles loaded");
    const int n = h->P.n;
    const SurfaceSizes sz = surface_sizes(n);
    if (!h->surf.sums) {
        SurfaceScratch z{};
        if ((st = dalloc_t(h, &z.bits, sz.bits)) != MPM_OK) return st;
        if ((st = dalloc_t(h, &z.counts, sz.words)) != MPM_OK) return st;
        if ((st = dalloc_t(h, &z.sums, sz.units + 1)) != MPM_OK) return st;
        h->surf = z;
    }
    const float4 *G = current_grid(h);
    const double dx = 1.0 / n;
    const float scale = (float)(1.0 / (h->env_rho[env] * dx * dx * dx));   // density / rho
    launch_surface_count(G, n, h->P.nb, h->nbe, (uint32_t)env, scale, iso, h->surf, h->elem_grid, h->stream);
    // device output needs no host-side total: the triangles follow at once, and the
    // total arrives with them
    if (on_device && max_tri > 0)
        launch_surface_emit(G, n, h->P.nb, h->nbe, (uint32_t)env, scale, iso, (float)dx, h->surf, tri,
                            (uint64_t)max_tri, h->stream);
    CK(cudaGetLastError());
    CK(cudaMemcpyAsync(h->h_total, h->surf.sums + sz.units, sizeof(uint32_t), cudaMemcpyDeviceToHost, h->stream));
    CK(cudaStreamSynchronize(h->stream));
    const uint32_t total = *h->h_total;
    *n_tri = total;
    const uint64_t nwrite = std::min<uint64_t>(total, (uint64_t)max_tri);
    if (nwrite == 0 || on_device) return MPM_OK;
    size_t cap = h->surf_tri_cap;
    if (cap < nwrite) {   // the old buffer stays with the handle until mpm_destroy
        if ((st = ensure(h, &h->surf_tri, &cap, 9 * (size_t)nwrite)) != MPM_OK) return st;
        h->surf_tri_cap = nwrite;
    }
    float *dst = h->surf_tri;
    launch_surface_emit(G, n, h->P.nb, h->nbe, (uint32_t)env, scale, iso, (float)dx, h->surf, dst, nwrite, h->stream);
    CK(cudaGetLastError());
    CK(cudaMemcpyAsync(tri, dst, sizeof(float) * 9 * nwrite, cudaMemcpyDeviceToHost, h->stream));
    CK(cudaStreamSynchronize(h->stream));
    return MPM_OK;
}

}  // extern "C"

// ================================================== asynchronous readback

extern "C" {

mpm_status mpm_read_particles_async(mpm_handle *h, float *x, float *v, float *F, float *C) {
    mpm_status st = check_handle(h);
    if (st != MPM_OK) return st;
    if (!h->loaded) return fail(MPM_ERR_STATE, "no particles loaded");
    const size_t N = (size_t)h->n;
    if (N == 0) return MPM_OK;
    if (!h->rb_stream) {
        CK(cudaStreamCreateWithFlags(&h->rb_stream, cudaStreamNonBlocking));
        for (int b = 0; b < 2; ++b) {
            CK(cudaEventCreateWithFlags(&h->rb_gathered[b], cudaEventDisableTiming));
            CK(cudaEventCreateWithFlags(&h->rb_copied[b], cudaEventDisableTiming));
        }
    }
    if (h->rb_cap < 24 * N) {   // a smaller earlier pair stays with the handle until mpm_destroy
        CK(cudaStreamSynchronize(h->rb_stream));
        for (int b = 0; b < 2; ++b)
            if ((st = dalloc_t(h, &h->rb_stage[b], 24 * N)) != MPM_OK) return st;
        h->rb_cap = 24 * N;
        h->rb_used[0] = h->rb_used[1] = false;
    }
    const int b = h->rb_next;
    h->rb_next ^= 1;
    // the copy two reads ago out of this staging buffer must be done before it is refilled
    if (h->rb_used[b]) CK(cudaStreamWaitEvent(h->stream, h->rb_copied[b], 0));
    float *sx = h->rb_stage[b], *sv = sx + 3 * N, *sF = sv + 3 * N, *sC = sF + 9 * N;
    launch_read_out(cur_state(h), h->fb.vc, (uint32_t)N, x ? sx : nullptr, v ? sv : nullptr, F ? sF : nullptr,
                    C ? sC : nullptr, h->elem_grid, h->stream);
    CK(cudaGetLastError());
    CK(cudaEventRecord(h->rb_gathered[b], h->stream));
    CK(cudaStreamWaitEvent(h->rb_stream, h->rb_gathered[b], 0));
    if (x) CK(cudaMemcpyAsync(x, sx, sizeof(float) * 3 * N, cudaMemcpyDeviceToHost, h->rb_stream));
    if (v) CK(cudaMemcpyAsync(v, sv, sizeof(float) * 3 * N, cudaMemcpyDeviceToHost, h->rb_stream));
    if (F) CK(cudaMemcpyAsync(F, sF, sizeof(float) * 9 * N, cudaMemcpyDeviceToHost, h->rb_stream));
    if (C) CK(cudaMemcpyAsync(C, sC, sizeof(float) * 9 * N, cudaMemcpyDeviceToHost, h->rb_stream));
    CK(cudaEventRecord(h->rb_copied[b], h->rb_stream));
    h->rb_used[b] = true;
    return MPM_OK;
}

mpm_status mpm_wait_read(mpm_handle *h) {
    mpm_status st = check_handle(h);
    if (st != MPM_OK) return st;
    if (h->rb_stream) CK(cudaStreamSynchronize(h->rb_stream));
    return poll_error(h, false);
}

}  // extern "C"
