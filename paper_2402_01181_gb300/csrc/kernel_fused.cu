// kernel_fused.cu -- one MLS-MPM sub-step as a single persistent kernel over
// the occupied 4x4x4-cell grid blocks.
//
// Sub-step k reads the grid G_k (mass, momentum after P2G of the particles at
// x_k) and the particles, grouped by the block of their stencil base, and
// writes x_{k+1}, F_{k+1} and the P2G of the new state into G_{k+1}:
//
//   per occupied block b (one CTA iteration):
//   1. grid operation (Eq. 7, gravity, tool contact Eqs. 11, 15-19, walls) of
//      the 6^3 nodes that the stencils of b's particles touch, into shared
//      memory;
//   2. per particle (passes of one particle per thread): G2P (Eqs. 8-9), F
//      update (Eq. 4), advection (Eq. 10), Kirchhoff stress of the new F
//      (Eqs. 5-6) and the affine momentum A = m C - dt V^0 (4/dx^2) tau;
//   3. a stable counting sort of the particles by their new block: every pass
//      writes its particles grouped by the direction (-1..1)^3 to their new
//      block and records where each group starts; the next sub-step's CTA for
//      block b' reads the runs heading to b' from its 27 neighbours, in
//      ascending source-block order;
//   4. P2G (Eqs. 1-3) of up to 2 passes of new particle states at a time into an
//      8^3-node shared arena around b.  The arena accumulates in 32-bit fixed
//      point with native shared integer atomics (shared float atomics are
//      several times slower): mass in units of m_p 2^-23, momentum in units of
//      B 2^-23 where B bounds every value that the group scatters (2^-22 in
//      groups of 1,024 and in recorded rollouts).  Weights are at most 0.42, so no contribution exceeds
//      2^22 and no node sum can overflow; the integer sums are exact, hence
//      independent of the order of the atomics.  A particle that moved further
//      than one cell scatters straight into G_{k+1} with float atomics instead.
//   5. the arena is converted back to floats and added to G_{k+1} with float4
//      atomics (only the 6^3 nodes around b when every base cell lies in b),
//      and the nodes read are returned to zero.
//
// G2P and P2G run their x/y (and z/mass) components on the packed f32x2 pipe.
//
// A launch does one sub-step, or several with a grid-wide wait between them.
//
// Grid buffers rotate over three slots (read G_k, write G_{k+1}, clear
// G_{k-1} for reuse), particle buffers and run tables over two, counters over
// three or four (a slot no CTA reads any more is zeroed meanwhile); the last CTA
// of a launch advances the sub-step index.
//
// Times in this file's comments are us per frame (25 sub-steps and the readout on the
// device) of the bodies of perf/cases.py under a moving tool: 2K patch, 8K cube, 30K and
// 200K slab, 1M and 8M block, one body each, both sides in turn on one GPU.  Other
// bodies and GPUs shift both sides by up to 15% (8K cube 399 to 467, 30K slab 337 to
// 376); lightly pressed ones are faster (30K slab 260).
#include <algorithm>
#include <climits>

#include "common.cuh"
#include "launch.h"

namespace gbmpm {

namespace {

constexpr int CMAX = kRunsShared;      // run candidates (source chunk x direction) per block in shared memory
// What a launch belongs to: plain stepping, or a recorded rollout (mpm_tape_record),
// whose sub-steps keep their records (kRecord) or not (kRollout).
enum Use { kStep, kRollout, kRecord };
// Fixed-point units per bound of a group of up to 512 or 1,024 particles: 2^23 or
// 2^22.  A weight is at most 0.75^3 = 0.42, so a term stays below 2^22 (kMagic's
// range) and a node's sum of all the group's terms below 2^31.  Rollouts keep 2^22
// and the bound about the stencil's base: the pose gradients of a rollout in contact
// hang on which nodes under the tool stick and which slide, and a rounding that
// every run shares moves them by more than one run differs from another (30K slab,
// 100 sub-steps: by 1.0e-4 of their norm with 2^23 and the bound about the centre,
// runs differ by 2.4e-5).
template <int GROUP, Use USE>
constexpr float kFixUnits = GROUP <= 512 && USE == kStep ? 8388608.0f : 4194304.0f;
constexpr float kMagic = 12582912.0f;   // 1.5 * 2^23: float -> nearest int for |v| < 2^22
// arena node (x, y, z) in [0,8)^3 sits at x + kAy y + kAz z: kAz = 68 keeps the
// bases of a z-pair of cells in distinct shared-memory banks
constexpr int kAy = 8, kAz = 68, kArena = 8 * kAz;

// Shared memory of a CTA of T threads that stages GP passes (GP T particles)
// per arena flush.
// PD: particle copies in flight per thread (a pass's particle is copied PD
// passes ahead of its use)
template <int T, int GP, int PD = 1>
struct FusedSmem {
    static constexpr int NW = T / 32;
    static constexpr int GROUP = GP * T;
    // double-buffered per-block inputs, prefetched with cp.async one block ahead:
    // the 6^3 grid nodes [4b, 4b+5]^3 (mass, momentum; turned into velocities
    // in place by the grid operation) and the block's inbox of incoming runs
    float4 graw[2][216];
    // the block's grid velocities as (x, y) and z, where shared memory has room (not
    // in configuration 2): a node of the gather costs 3 wavefronts of the busiest
    // unit instead of the 4 of a 16-byte word, and fewer conflicts (8K cube 417 -> 399
    // us a frame, 200K slab 629 -> 604, 1M particles 2289 -> 2267)
    static constexpr bool kSplit = !(T == 128 && GP == 2);
    float2 vxy[kSplit ? 216 : 1];
    float vz[kSplit ? 216 : 1];
    uint4 inbox[2][kInbox];
    EnvParams ep[2];               // the block's environment: material
    ToolFrame tools[2][kMaxTools]; // and its tool frames for this sub-step
    uint32_t items[2], bids[2];    // work items (their place in the lists) and their blocks (kNoBlock: none)
    uint32_t own;                  // a block that this CTA keeps for the launch's next sub-step, or kNoBlock
    int acc[4][kArena];            // P2G arena over nodes [4b-1, 4b+6]^3 (fixed point, padded strides)
    // staged P2G inputs of one group: f (3) and the arena base, q (3) and A dx (9) of
    // each particle as four 16-byte words, swizzled (st) so that the words of any 8
    // neighbouring slots lie in distinct banks: the scatter reads slots in bank order
    // of their bases, at random, and the shared-memory pipe is the busiest unit (58%);
    // as 16 separate words 1M particles took 2303 us a frame, now 2258
    float4 st4[4 * GROUP];
    static __device__ __forceinline__ int st(int slot, int word) { return 4 * slot + (word ^ ((slot >> 1) & 3)); }
    // the group's particles bucketed by the shared-memory bank of their arena
    // base: rank within the bucket (and the bucket) per slot (kOut: not in the
    // arena), bucket sizes, and the slots in bucket order
    static constexpr uint16_t kOut = 0xffffu;
    uint16_t st_key[GROUP];
    uint16_t order[GROUP];
    uint32_t ccount[32];
    // each thread's particle of the current pass, prefetched with cp.async a pass
    // ahead (a thread reads and refills only its own slot)
    float4 pxi[PD][T], pf0[PD][T], pf1[PD][T];
    float pf2[PD][T];
    uint32_t cand_start[CMAX];     // first slot of each run
    uint32_t cand_pre[CMAX];       // exclusive prefix of run lengths
    uint32_t lane_first[27], lane_off[27];
    // per pass parity: per direction, each warp's count of it (one byte per
    // warp, so that a lane sums all warps' counts of its direction in one load)
    static constexpr int NWP = NW <= 4 ? 4 : NW;
    alignas(16) uint8_t wcnt[2][28][NWP];
    uint32_t ncand, total, out_base, chunk_first, npass, mask, bmax, wide;
    uint32_t nact, nheavy;         // active blocks, heavy ones among them
    uint32_t m3;                   // sub-step index mod 3
    StepRecord rec;                // the sub-step's record (recording sub-steps)
    bool go;                       // the launch's next sub-step may start
};

// resident CTAs per SM for which a configuration is compiled: 228 KB of shared
// memory per SM with 1 KB reserved per CTA, 64 K registers
template <int T, int GP>
constexpr int kMinBlocks = T == 512 ? 1 : T == 256 ? 3 : (GP == 1 ? 5 : 4);
static_assert(3 * (sizeof(FusedSmem<256, 2>) + 1024) <= 228 * 1024, "shared memory for three CTAs per SM");
static_assert(4 * (sizeof(FusedSmem<128, 2>) + 1024) <= 228 * 1024, "shared memory for four CTAs per SM");
static_assert(5 * (sizeof(FusedSmem<128, 1>) + 1024) <= 228 * 1024, "shared memory for five CTAs per SM");
static_assert(4 * (sizeof(FusedSmem<128, 2, 2>) + 1024) <= 228 * 1024, "configuration 2: four CTAs per SM");
static_assert(2 * (sizeof(FusedSmem<256, 2, 2>) + 1024) <= 228 * 1024, "configuration 4: two CTAs per SM");

// the record k sub-steps after r
__host__ __device__ __forceinline__ StepRecord record_of(StepRecord r, uint32_t k) {
    const size_t f = k * r.floats, w = k * r.words, g = k * r.nodes;
    r.xi += f / 4; r.f0 += f / 4; r.f1 += f / 4; r.f2 += f; r.src += f;
    r.vc.vc0 += f / 4; r.vc.vc1 += f / 4; r.vc.vc2 += f / 4;
    r.blk += w / 2; r.act += w; r.nact += w;
    r.grid += g; r.vgrid += g;
    return r;
}

__device__ __forceinline__ BlockTab load_tab(const BlockTab *p) {
    const uint4 v = __ldcg(reinterpret_cast<const uint4 *>(p));
    BlockTab t;
    t.stamp = v.x; t.first = v.y; t.npass = v.z; t.pad = v.w;
    return t;
}

__device__ __forceinline__ int dir_dx(int d) { return d % 3 - 1; }
__device__ __forceinline__ int dir_dy(int d) { return (d / 3) % 3 - 1; }
__device__ __forceinline__ int dir_dz(int d) { return d / 9 - 1; }

// list grid block g among those to clear of G_{stamp}, kept in list slot stamp mod 3
__device__ __forceinline__ void mark_clear(const FusedBufs &B, uint32_t g, uint32_t stamp, int slot) {
    if (atomicExch(&B.gstamp[g], stamp) != stamp) B.clist[slot][atomicAdd(&B.ctrl->nclear[stamp & 3u], 1u)] = g;
}

// nearest integer of v (|v| < 2^22) via the float mantissa
__device__ __forceinline__ int fix_round(float scaled_plus_magic) {
    return __float_as_int(scaled_plus_magic) - 0x4B400000;
}

// G[addr] += v as one vector reduction (no value returned)
__device__ __forceinline__ void red_add4(float4 *addr, float4 v) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem, bool valid) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem);
    const int bytes = valid ? 16 : 0;   // 0: fill with zeros, read nothing
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(gmem), "r"(bytes) : "memory");
}
// 16 bytes into shared memory without allocating in L1 (streamed particle state)
__device__ __forceinline__ void cp_async16_cg(void *smem, const void *gmem) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async4(void *smem, const void *gmem) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_but_one() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_but_two() { asm volatile("cp.async.wait_group 2;\n" ::: "memory"); }

// Slot of logical index j among the block's incoming runs (binary search of
// the runs' exclusive prefix).  This CTA's part of FusedBufs::runs holds them
// (prefix, first slot) where they are more than CMAX.
template <bool MORE, class Smem>
__device__ __forceinline__ uint32_t source_slot(const Smem &s, const FusedBufs &B, uint32_t ncand, uint32_t j) {
    if (MORE && ncand > CMAX) {
        const uint2 *runs = B.runs + (size_t)blockIdx.x * kRunsListed;
        uint32_t lo = 0, hi = ncand - 1u;
        while (lo < hi) {
            const uint32_t mid = (lo + hi + 1u) >> 1;
            if (__ldcg(&runs[mid].x) <= j) lo = mid; else hi = mid - 1u;
        }
        const uint2 r = __ldcg(&runs[lo]);
        return r.y + (j - r.x);
    }
    int lo = 0, hi = (int)ncand - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (s.cand_pre[mid] <= j) lo = mid; else hi = mid - 1;
    }
    return s.cand_start[lo] + (j - s.cand_pre[lo]);
}

// Start copying the particle with logical index j into this thread's slot.
template <bool MORE, class Smem>
__device__ __forceinline__ void prefetch_particle(Smem &s, const FusedBufs &B, uint32_t in_off, uint32_t ncand,
                                                  uint32_t j, int tid, int set) {
    const uint32_t src = in_off + source_slot<MORE>(s, B, ncand, j);
    cp_async16_cg(&s.pxi[set][tid], &B.P[0].xi[src]);
    cp_async16_cg(&s.pf0[set][tid], &B.P[0].f0[src]);
    cp_async16_cg(&s.pf1[set][tid], &B.P[0].f1[src]);
    cp_async4(&s.pf2[set][tid], &B.P[0].f2[src]);
}

// Start copying global block b's grid region of G_k, its inbox, and its
// environment's material and tool frames into buffer buf.
template <int T, class Smem>
__device__ __forceinline__ void prefetch_block(Smem &s, int buf, uint32_t b, const uint4 *__restrict__ inbox,
                                               const float4 *__restrict__ Gcur, const DevParams &P,
                                               const ToolFrame *__restrict__ tools, int tid) {
    const int nb = P.nb, n = P.n;
    const uint32_t e = b >> (3 * P.lnb);
    int bx, by, bz;
    block_coords(b, P.lnb, bx, by, bz);
    constexpr int kTw = (int)(sizeof(ToolFrame) / 16);   // 16-byte words per frame
    const int ntw = P.tstride * kTw;
    for (int q = tid; q < 216 + kInbox + 2 + ntw; q += T) {
        if (q < 216) {
            const int i = 4 * bx + q % 6, j = 4 * by + (q / 6) % 6, k = 4 * bz + q / 36;
            const bool ok = i < n && j < n && k < n;
            cp_async16(&s.graw[buf][q], ok ? (const void *)&Gcur[node_addr_env(e, i, j, k, nb, P.nbe)] : (const void *)Gcur,
                       ok);
        } else if (q < 216 + kInbox) {
            const int x = q - 216;
            cp_async16(&s.inbox[buf][x], &inbox[(size_t)b * kInbox + x], true);
        } else if (q < 216 + kInbox + 2) {
            const int x = q - 216 - kInbox;
            cp_async16(reinterpret_cast<uint4 *>(&s.ep[buf]) + x, reinterpret_cast<const uint4 *>(&P.envp[e]) + x, true);
        } else {
            const int x = q - 216 - kInbox - 2;
            cp_async16(reinterpret_cast<uint4 *>(&s.tools[buf][0]) + x,
                       reinterpret_cast<const uint4 *>(tools + (size_t)e * P.tstride) + x, true);
        }
    }
    cp_async_commit();
}


// The two configurations between which the host chooses by the blocks in use (512
// threads, and 256 with 2 CTAs per SM): they report them, and obey a LaunchGate.
template <int MINB, Use USE>
constexpr bool kGated = MINB <= 2 && USE == kStep;

// MINB: resident CTAs per SM the configuration is compiled for (the register budget)
// MORE: a block's runs beyond CMAX are listed in FusedBufs::runs.  CTAs of 128 threads
// write more, smaller runs; with them a block takes in as many particles as with
// 256.  (An instantiation of its own, for environments that can need it: the test
// in every particle's copy made 256 environments of 5K to 40K 1.6% slower.)
// USE kRecord: also write, for the reverse mode, every block's input particles at
// their output positions (inside the range [out_base, out_base + total) the
// block's output was allocated) with their input positions, the list of
// blocks in work order with each one's range, the list's length, and the grid
// of each block's region before and after the grid operation.
// One sub-step.  first: the launch's first (the arena is cleared then); last: the
// launch's last (WRITE_VC: the one that writes v and C).  target: CTAs of the
// launch times its sub-steps up to this one.  Returns whether to go on: false
// after the last sub-step, or when the wait for the other CTAs ran out.
template <bool WRITE_VC, int T, int GP, int MINB, Use USE, int PD, bool MORE>
__device__ __forceinline__ bool fused_substep(FusedSmem<T, GP, PD> &s, const DevParams &P, const FusedBufs &B,
                                              const ToolFrame *__restrict__ tools, const StepRecord &rec0, uint32_t k,
                                              uint32_t step, uint32_t target, bool first, bool last) {
    using Smem = FusedSmem<T, GP, PD>;
    static_assert(PD == 1 || PD == 2, "one or two particle copies in flight");
    constexpr int NW = Smem::NW, GROUP = Smem::GROUP;
    constexpr bool RECORD = USE == kRecord;
    constexpr float kFix = kFixUnits<GROUP, USE>;
    constexpr bool kEarly = T * MINB <= 512, kKeep = MINB == 1;
    // Particles over which a block is heavy: one pass of the CTA.  With two CTAs per SM
    // a scene has about a block per CTA, and half a pass tells a full block of a sparse
    // slab from one at its edge: CTA i and the one a wave later, which share an SM,
    // then take one of each (30K slab 368 -> 340 us a frame in contact).
    constexpr uint32_t kHeavy = MINB == 2 ? T / 2 : T;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    Ctrl *ctrl = B.ctrl;
    const int par = step & 1, m3 = step % 3;
    const int m3n = (m3 + 1) % 3, m3c = (m3 + 2) % 3;
    // the two buffers of each array lie in one allocation: the sub-step's parity
    // is an index offset, the bases stay kernel parameters
    const uint32_t in_off = par ? B.pstride : 0u, out_off = B.pstride - in_off;            // particle slots
    const uint32_t chunk_in = par ? B.cstride : 0u, chunk_out = B.cstride - chunk_in;      // chunks
    const uint32_t blk_in = par ? B.nblocks : 0u, blk_out = B.nblocks - blk_in;            // per-block tables
    const float4 *__restrict__ Gcur = B.G[m3];
    float4 *Gnext = B.G[m3n];
    float4 *Gclr = B.G[m3c];
    // the active blocks: heavy ones listed from the front, light ones from the
    // back, and handed out heavy first so that the launch ends on short items
    const unsigned long long nhl = *(volatile unsigned long long *)&ctrl->nactive[m3][0];
    const uint32_t nheavy = (uint32_t)nhl, nact = (uint32_t)nhl + (uint32_t)(nhl >> 32);
    const uint32_t acap = B.nblocks;
    auto item_block = [&](uint32_t it) -> uint32_t {
        return it >= s.nact ? kNoBlock : __ldcg(&B.alist[0][blk_in + (it < s.nheavy ? it : acap - 1u - (it - s.nheavy))]);
    };
    const uint32_t nclr = *(volatile uint32_t *)&ctrl->nclear[(step + 3u) & 3u];     // G_{k-1}'s
    const uint32_t *__restrict__ clr = B.clist[m3c];
    const uint32_t nparticles = ctrl->n_particles;
    const uint32_t nchunk_cap = B.nblocks + nparticles / T + 1;
    const int nb = P.nb, n = P.n;
    const uint32_t nbe = P.nbe;
    uint32_t err = 0;

    // prologue: this CTA's first block and its inputs.  With one CTA per SM (kKeep)
    // that is, after the launch's first sub-step, the block it kept, known without a
    // memory access, so that its inputs are under way before the lists' sizes
    // arrive; the lists then hold the blocks that no CTA kept (8K cube 444 -> 424 us a
    // frame, 2K patch 109 -> 106; with two CTAs per SM a fixed placement loses more
    // where two heavy blocks share an SM: the 30K slab's reset 408 -> 438).  Otherwise
    // the first gridDim.x items are the front of the heavy list, then the light
    // list's, each CTA's at a place that does not depend on the lists' sizes: both
    // entries are read together with the sizes.  The shared counter hands out the rest.
    const bool lists = !kKeep || first;
    const uint32_t fixed = lists ? gridDim.x : 0u;     // items that the counter starts from
    const StepRecord &rec = s.rec;
    if (RECORD && tid == 0) s.rec = record_of(rec0, k);
    if (tid == T - 1) {
        uint32_t item = 0, b;
        if (lists) {
            const uint32_t back = gridDim.x - 1u - blockIdx.x;     // this CTA's place in the light list
            const uint32_t *al = B.alist[0] + blk_in;
            const uint32_t hb = blockIdx.x < acap ? __ldcg(&al[blockIdx.x]) : 0u;
            const uint32_t lb = back < acap ? __ldcg(&al[acap - 1u - back]) : 0u;
            const bool heavy = blockIdx.x < nheavy;
            item = heavy ? blockIdx.x : nheavy + back;
            b = item >= nact ? kNoBlock : heavy ? hb : lb;
        } else {
            b = s.own;
            if (b == kNoBlock && nact > 0u) {
                item = atomicAdd(&ctrl->work[m3], 1u);
                if (item < nact)
                    b = __ldcg(&B.alist[0][blk_in + (item < nheavy ? item : acap - 1u - (item - nheavy))]);
            }
        }
        s.items[0] = item;
        s.bids[0] = b;
        s.own = kNoBlock;
    }
    __syncthreads();
    if (s.bids[0] != kNoBlock) prefetch_block<T>(s, 0, s.bids[0], blk_in ? B.inbox[1] : B.inbox[0], Gcur, P, tools, tid);
    if (tid == 0) { s.m3 = (uint32_t)m3; s.nact = nact; s.nheavy = nheavy; }
    // the P2G arena starts at zero; every flush returns the nodes it read to zero
    if (first)
        for (int q = tid; q < 4 * kArena; q += T) (&s.acc[0][0])[q] = 0;
    // 0. while the first block's inputs land: clear the grid blocks G_{k-1} touched,
    //    so that sub-step k+1 can scatter into it (a different buffer from G_k)
    for (uint32_t q = blockIdx.x * T + tid; q < nclr * 64u; q += gridDim.x * T)
        Gclr[__ldcg(&clr[q >> 6]) * 64u + (q & 63u)] = make_float4(0.f, 0.f, 0.f, 0.f);
    // the counters that the next sub-step takes, idle since the last one but one
    if (blockIdx.x == gridDim.x - 1 && tid == 0) {
        if (!first && *(volatile uint32_t *)&ctrl->part_alloc[m3c] != nparticles) err |= kErrCapacity;
        ctrl->work[m3n] = 0;
        ctrl->part_alloc[m3n] = 0;
        ctrl->chunk_alloc[m3n] = 0;
        ctrl->nactive[m3c][0] = 0;
        ctrl->nactive[m3c][1] = 0;
        ctrl->nclear[(step + 2u) & 3u] = 0;
        if (RECORD) *rec.nact = nact;
    }
    cp_async_wait_all();
    __syncthreads();

    for (int cb = 0;; cb ^= 1) {
        const uint32_t b = s.bids[cb];                 // global block
        if (b == kNoBlock) break;
        if (RECORD && tid == 0) rec.act[s.items[cb]] = b;
        const uint32_t env = b >> (3 * P.lnb);          // environment
        const uint32_t eb0 = env * nbe;                 // its first global block
        int bx, by, bz;
        block_coords(b, P.lnb, bx, by, bz);
        const EnvParams &ep = s.ep[cb];
        const float m = ep.mass;
        // the next work item, unless the lists hold none: the atomic is issued here and
        // its result is consumed after this thread's share of the grid operation
        uint32_t next_item = s.nact;
        if (tid == T - 1 && s.nact > fixed) next_item = fixed + atomicAdd(&ctrl->work[s.m3], 1u);
        uint32_t alloc_ob = 0, alloc_cf = 0;     // thread 0: the block's output range and chunks
        float4 *gv = s.graw[cb];

        // 1. grid operation of the 6^3 G2P region, in place (warps 1 ..)
        for (int q = tid - 32; q >= 0 && q < 216; q += T - 32) {
            const int i = 4 * bx + q % 6, j = 4 * by + (q / 6) % 6, k = 4 * bz + q / 36;
            const float4 g = gv[q];
            float3 v = make_float3(0.f, 0.f, 0.f);
            if (i < n && j < n && k < n) v = grid_node_update(g.x, g.y, g.z, g.w, i, j, k, P, s.tools[cb], ep.ntools);
            if (Smem::kSplit) {
                s.vxy[q] = make_float2(v.x, v.y);
                s.vz[q] = v.z;
            } else {
                gv[q] = make_float4(v.x, v.y, v.z, 0.f);
            }
            if (RECORD && i < n && j < n && k < n) {
                const uint32_t a = node_addr_env(env, i, j, k, nb, nbe);
                rec.grid[a] = g;
                rec.vgrid[a] = make_float4(v.x, v.y, v.z, 0.f);
            }
        }
        if (tid < 32) s.ccount[tid] = 0u;
        for (int q = tid; q < 2 * 28 * Smem::NWP / 4; q += T) reinterpret_cast<uint32_t *>(&s.wcnt[0][0][0])[q] = 0u;
        if (tid == T - 1) {
            s.items[cb ^ 1] = next_item;
            s.bids[cb ^ 1] = item_block(next_item);
        }
        // 2. warp 0: the runs heading to b, in ascending source-block order
        //    (direction d = 26 .. 0, source pass 0 .. 3), with their exclusive
        //    prefix = logical index of each run's first particle
        if (warp == 0) {
            const uint4 *ib = s.inbox[cb];
            uint32_t nc = 0, carry = 0;
            if (ib[kInbox - 1].x != step) {
                // lane l takes direction 26 - l, all its source passes: one scan
                uint32_t start[kNpMax], cnt[kNpMax], sum = 0, pos = 0;
#pragma unroll
                for (int p = 0; p < kNpMax; ++p) {
                    uint4 e = make_uint4(0u, 0u, 0u, 0u);
                    if (lane < 27) e = ib[(26 - lane) * kNpMax + p];
                    const bool ok = e.z == step && e.y > 0u;     // step >= 1
                    const unsigned bal = __ballot_sync(0xffffffffu, ok);
                    start[p] = e.x;
                    cnt[p] = ok ? e.y : 0u;
                    sum += cnt[p];
                    pos += __popc(bal & ((1u << lane) - 1u));
                    nc += __popc(bal);
                }
                uint32_t incl = sum;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                carry = __shfl_sync(0xffffffffu, incl, 31);
                uint32_t pre = incl - sum;
#pragma unroll
                for (int p = 0; p < kNpMax; ++p)
                    if (cnt[p] > 0u) {
                        s.cand_start[pos] = start[p];
                        s.cand_pre[pos] = pre;
                        ++pos;
                        pre += cnt[p];
                    }
            } else {
                // a source wrote more passes than the inbox holds: walk its run tables
                uint32_t np = 0, first = 0;
                if (lane < 27) {
                    const int d = 26 - lane;
                    const int sx = bx - dir_dx(d), sy = by - dir_dy(d), sz = bz - dir_dz(d);
                    if (sx >= 0 && sy >= 0 && sz >= 0 && sx < nb && sy < nb && sz < nb) {
                        const BlockTab t = load_tab(&B.tabs[0][blk_in + eb0 + block_id(sx, sy, sz, nb)]);
                        if (t.stamp == step) { np = t.npass; first = t.first; }
                    }
                }
                uint32_t incl = np;
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                if (lane < 27) { s.lane_first[lane] = first; s.lane_off[lane] = incl - np; }
                uint32_t ncand = __shfl_sync(0xffffffffu, incl, 26);
                constexpr uint32_t most = MORE ? kRunsListed : CMAX;
                if (ncand > most) { ncand = most; err |= kErrCapacity; }
                __syncwarp();
                for (uint32_t c0 = 0; c0 < ncand; c0 += 32) {
                    const uint32_t c = c0 + lane;
                    uint2 r = make_uint2(0u, 0u);
                    if (c < ncand) {
                        int l = 0;
                        while (l < 26 && s.lane_off[l + 1] <= c) ++l;
                        r = __ldcg(&B.chunks[0][chunk_in + s.lane_first[l] + (c - s.lane_off[l])].run[26 - l]);
                    }
                    uint32_t incl2 = r.y;
                    for (int o = 1; o < 32; o <<= 1) {
                        const uint32_t y = __shfl_up_sync(0xffffffffu, incl2, o);
                        if (lane >= o) incl2 += y;
                    }
                    if (MORE && ncand > CMAX) {
                        if (c < ncand) B.runs[(size_t)blockIdx.x * kRunsListed + c] = make_uint2(carry + incl2 - r.y, r.x);
                    } else if (c < ncand) {
                        s.cand_start[c] = r.x;
                        s.cand_pre[c] = carry + incl2 - r.y;
                    }
                    carry += __shfl_sync(0xffffffffu, incl2, 31);
                }
                nc = ncand;
            }
            __syncwarp();
            if (lane == 0) {
                s.ncand = nc;
                s.total = carry;
                s.npass = (carry + T - 1) / T;
                // issued here, consumed after the barrier below
                alloc_ob = atomicAdd(&ctrl->part_alloc[s.m3], carry);
                alloc_cf = atomicAdd(&ctrl->chunk_alloc[s.m3], (carry + T - 1) / T);
                s.mask = 0;
                s.bmax = 0;
                s.wide = 0;
            }
        }
        __syncthreads();
        const uint32_t ncand = s.ncand;
        const uint32_t total = s.total, npass = s.npass;
        // thread 0: the block's table for the next sub-step and its output range,
        // read by every thread after the first pass's barrier; if the allocation
        // overflowed, the range starts past the end of the particle and chunk
        // arrays and nothing is written
        if (tid == 0) {
            BlockTab t;
            t.pad = 0;
            const bool fit = alloc_ob + total <= nparticles && alloc_cf + npass <= nchunk_cap;
            if (fit) {
                t.stamp = step + 1; t.first = alloc_cf; t.npass = npass;
            } else {
                err |= kErrCapacity;
                t.stamp = 0; t.first = 0; t.npass = 0;
            }
            B.tabs[0][blk_out + b] = t;
            if (RECORD) rec.blk[s.items[cb]] = make_uint2(fit ? alloc_ob : 0u, fit ? total : 0u);
            s.out_base = fit ? alloc_ob : nparticles;
            s.chunk_first = fit ? alloc_cf : nchunk_cap;
        }
        // this thread's particle of the first pass, then the next block's inputs;
        // both land while this block computes
        if (npass > 0 && (uint32_t)tid < total) prefetch_particle<MORE>(s, B, in_off, ncand, (uint32_t)tid, tid, 0);
        cp_async_commit();
        if (PD == 2) {   // and the second pass's
            if (npass > 1 && (uint32_t)(T + tid) < total) prefetch_particle<MORE>(s, B, in_off, ncand, (uint32_t)(T + tid), tid, 1);
            cp_async_commit();
        }
        if (s.bids[cb ^ 1] != kNoBlock) prefetch_block<T>(s, cb ^ 1, s.bids[cb ^ 1], blk_in ? B.inbox[1] : B.inbox[0], Gcur, P, tools, tid);
        else cp_async_commit();
        const int ox = 4 * bx - 1, oy = 4 * by - 1, oz = 4 * bz - 1;   // arena origin

        // Blocks of the next sub-step (the last warp) and grid blocks to clear before
        // G_{k+1}'s reuse (the one before it): two chains of dependent global atomics.
        // Where registers allow (kEarly) the stamps are exchanged before the last
        // scatter and the lists appended to after the last flush, so that the first
        // round trip is off the block's chain; otherwise both run after the block,
        // beside warp 0's set-up of the next one.
        uint32_t mark_b = 0, mark_old = step + 1;
        auto mark_begin = [&](uint32_t mask) {
            if (warp < NW - 2 || lane >= 27) return;
            const int tx = bx + dir_dx(lane), ty = by + dir_dy(lane), tz = bz + dir_dz(lane);
            if (tx < 0 || ty < 0 || tz < 0 || tx >= nb || ty >= nb || tz >= nb) return;
            mark_b = eb0 + block_id(tx, ty, tz, nb);
            if (warp == NW - 2) mark_old = atomicExch(&B.gstamp[mark_b], step + 1);
            else if ((mask >> lane) & 1u) mark_old = atomicExch(&B.astamp[mark_b], step + 1);
        };
        auto mark_end = [&]() {
            if (mark_old == step + 1) return;
            if (warp == NW - 2) {
                B.clist[(step + 1u) % 3u][atomicAdd(&ctrl->nclear[(step + 1) & 3u], 1u)] = mark_b;
            } else {
                // kKeep: b itself (lane 13) stays with this CTA if it keeps no other; into
                // the lists goes the rest.  Heavy: b with more than kHeavy particles now.  A
                // neighbour's mark wins only for blocks that particles
                // enter from outside, which are light.
                if (kKeep && !last && lane == 13 && s.own == kNoBlock)
                    s.own = mark_b;
                else if (lane == 13 && total > kHeavy)
                    B.alist[0][blk_out + atomicAdd(&ctrl->nactive[s.m3 == 2u ? 0u : s.m3 + 1u][0], 1u)] = mark_b;
                else
                    B.alist[0][blk_out + acap - 1u - atomicAdd(&ctrl->nactive[s.m3 == 2u ? 0u : s.m3 + 1u][1], 1u)] = mark_b;
            }
        };
        for (uint32_t pass = 0; pass < npass; ++pass) {
            const uint32_t j = pass * T + tid;
            const bool valid = j < total;
            const int slot = (pass % GP) * T + tid;    // staging slot within the group
            int d = 31;
            uint32_t bound = 0u;      // this particle's share of the group bound (float bits)
            float nxp = 0.f, nyp = 0.f, nzp = 0.f, idf = 0.f, Fn[9], Cm[9], vx = 0.f, vy = 0.f, vz = 0.f;
            // this pass's particle is in the slot; the next block's inputs may still be landing
            // every thread commits, in order: pass 0's particle, [PD = 2: pass 1's
            // particle,] the next block's inputs, then one group per pass holding
            // the particle of pass + PD.  Wait for this pass's particle only.
            if (PD == 1) {
                if (pass == 0) cp_async_wait_but_one(); else cp_async_wait_all();
            } else {
                if (pass <= 1) cp_async_wait_but_two(); else cp_async_wait_but_one();
            }
            float4 xi = make_float4(0.f, 0.f, 0.f, 0.f), a0 = xi, a1 = xi;
            float f2 = 0.f;
            const int ps = (int)(pass % PD);   // slot set of this pass's particle
            if (valid) { xi = s.pxi[ps][tid]; a0 = s.pf0[ps][tid]; a1 = s.pf1[ps][tid]; f2 = s.pf2[ps][tid]; }
            const uint32_t jn = j + PD * T;
            if (valid) {
                const float F[9] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w, f2};
                idf = xi.w;
                // --- G2P from the shared velocities (Eqs. 8-9)
                int gx, gy, gz;
                const float fx = stencil_axis(xi.x, P.inv_dx, n, gx, err);
                const float fy = stencil_axis(xi.y, P.inv_dx, n, gy, err);
                const float fz = stencil_axis(xi.z, P.inv_dx, n, gz, err);
                int lx = gx - 4 * bx, ly = gy - 4 * by, lz = gz - 4 * bz;
                if (lx < 0 || lx > 3 || ly < 0 || ly > 3 || lz < 0 || lz > 3) {
                    err |= kErrCfl;
                    lx = min(max(lx, 0), 3); ly = min(max(ly, 0), 3); lz = min(max(lz, 0), 3);
                }
                float wx[3], wy[3], wz[3];
                bspline_weights(fx, wx);
                bspline_weights(fy, wy);
                bspline_weights(fz, wz);
                // With the stencil offset o = (ii, jj, kk) - f (cell units), the
                // affine sum of Eq. 9 is sum w v o^T = sum w v (ii, jj, kk)^T - v f^T:
                // the moments about the stencil base need no per-node offset and
                // vanish on the ii = 0 (jj = 0, kk = 0) layers.  The x and y
                // components run on the packed f32x2 pipe.
                const float2 w0 = make_float2(wx[0], wx[0]), w1 = make_float2(wx[1], wx[1]);
                const float2 w2 = make_float2(wx[2], wx[2]), w2d = make_float2(2.f * wx[2], 2.f * wx[2]);
                float2 vxy = make_float2(0.f, 0.f), mxy = vxy, myy = vxy, mzy = vxy;   // v, and moments along x, y, z
                float vzz = 0.f, mxz = 0.f, myz = 0.f, mzz = 0.f;
#pragma unroll
                for (int kk = 0; kk < 3; ++kk) {
#pragma unroll
                    for (int jj = 0; jj < 3; ++jj) {
                        const float wjk = wy[jj] * wz[kk];
                        const float2 wjk2 = make_float2(wjk, wjk);
                        const int r = lx + 6 * (ly + jj) + 36 * (lz + kk);
                        float2 h0, h1, h2;
                        float z0, z1, z2;
                        if (Smem::kSplit) {
                            h0 = s.vxy[r]; h1 = s.vxy[r + 1]; h2 = s.vxy[r + 2];
                            z0 = s.vz[r]; z1 = s.vz[r + 1]; z2 = s.vz[r + 2];
                        } else {
                            const float4 g0 = gv[r], g1 = gv[r + 1], g2 = gv[r + 2];
                            h0 = make_float2(g0.x, g0.y); h1 = make_float2(g1.x, g1.y); h2 = make_float2(g2.x, g2.y);
                            z0 = g0.z; z1 = g1.z; z2 = g2.z;
                        }
                        // a = sum_ii wx g, b = sum_ii ii wx g along the row
                        float2 axy = __fmul2_rn(w0, h0);
                        axy = __ffma2_rn(w1, h1, axy);
                        axy = __ffma2_rn(w2, h2, axy);
                        const float az = fmaf(wx[2], z2, fmaf(wx[1], z1, wx[0] * z0));
                        const float2 bxy = __ffma2_rn(w2d, h2, __fmul2_rn(w1, h1));
                        const float bz = fmaf(w2d.x, z2, wx[1] * z1);
                        vxy = __ffma2_rn(wjk2, axy, vxy);
                        vzz = fmaf(wjk, az, vzz);
                        mxy = __ffma2_rn(wjk2, bxy, mxy);
                        mxz = fmaf(wjk, bz, mxz);
                        if (jj > 0) {
                            const float2 s2 = jj == 1 ? wjk2 : __fadd2_rn(wjk2, wjk2);
                            myy = __ffma2_rn(s2, axy, myy);
                            myz = fmaf(s2.x, az, myz);
                        }
                        if (kk > 0) {
                            const float2 s2 = kk == 1 ? wjk2 : __fadd2_rn(wjk2, wjk2);
                            mzy = __ffma2_rn(s2, axy, mzy);
                            mzz = fmaf(s2.x, az, mzz);
                        }
                    }
                }
                vx = vxy.x; vy = vxy.y; vz = vzz;
                // C = (4 / dx^2) sum w v (x_i - x_p)^T = (4 / dx) (moments - v f^T)   (Eq. 9)
                const float cs = 4.0f * P.inv_dx;
                const float2 cxy = __ffma2_rn(make_float2(-fx, -fx), vxy, mxy);
                const float2 cyy = __ffma2_rn(make_float2(-fy, -fy), vxy, myy);
                const float2 czy = __ffma2_rn(make_float2(-fz, -fz), vxy, mzy);
                Cm[0] = cs * cxy.x; Cm[1] = cs * cyy.x; Cm[2] = cs * czy.x;
                Cm[3] = cs * cxy.y; Cm[4] = cs * cyy.y; Cm[5] = cs * czy.y;
                Cm[6] = cs * fmaf(-fx, vzz, mxz); Cm[7] = cs * fmaf(-fy, vzz, myz); Cm[8] = cs * fmaf(-fz, vzz, mzz);
                // --- Eq. 4 and Eq. 10
#pragma unroll
                for (int r = 0; r < 3; ++r)
#pragma unroll
                    for (int c = 0; c < 3; ++c)
                        Fn[3 * r + c] = F[3 * r + c] + P.dt * (Cm[3 * r] * F[c] + Cm[3 * r + 1] * F[3 + c] + Cm[3 * r + 2] * F[6 + c]);
                nxp = xi.x + P.dt * vx;
                nyp = xi.y + P.dt * vy;
                nzp = xi.z + P.dt * vz;
                // every value read from the slot has been consumed: refill it with the
                // next pass's particle
                if (pass + PD < npass && jn < total) prefetch_particle<MORE>(s, B, in_off, ncand, jn, tid, ps);
                if (!finite3(nxp, nyp, nzp)) {
                    err |= kErrNumeric;
                    nxp = xi.x; nyp = xi.y; nzp = xi.z;
                }
                // --- stress of the new state (Eqs. 5-6) and the P2G inputs (Eqs. 1-3)
                float t[6];
                kirchhoff(Fn, ep.mu, ep.lam, t, err);
                const float kst = ep.stress_k, dxs = P.dx;
                float A[9] = {(m * Cm[0] - kst * t[0]) * dxs, (m * Cm[1] - kst * t[1]) * dxs, (m * Cm[2] - kst * t[2]) * dxs,
                              (m * Cm[3] - kst * t[1]) * dxs, (m * Cm[4] - kst * t[3]) * dxs, (m * Cm[5] - kst * t[4]) * dxs,
                              (m * Cm[6] - kst * t[2]) * dxs, (m * Cm[7] - kst * t[4]) * dxs, (m * Cm[8] - kst * t[5]) * dxs};
                int hx, hy, hz;
                const float ex = stencil_axis(nxp, P.inv_dx, n, hx, err);
                const float ey = stencil_axis(nyp, P.inv_dx, n, hy, err);
                const float ez = stencil_axis(nzp, P.inv_dx, n, hz, err);
                // q = m v - A' fx: the value at stencil offset o is q + A' o
                const float qx = m * vx - (A[0] * ex + A[1] * ey + A[2] * ez);
                const float qy = m * vy - (A[3] * ex + A[4] * ey + A[5] * ez);
                const float qz = m * vz - (A[6] * ex + A[7] * ey + A[8] * ez);
                if (!(isfinite(qx) && isfinite(qy) && isfinite(qz))) err |= kErrNumeric;
                const int ax0 = hx - ox, ay0 = hy - oy, az0 = hz - oz;
                const bool in_arena = ax0 >= 0 && ax0 <= 5 && ay0 >= 0 && ay0 <= 5 && az0 >= 0 && az0 <= 5;
                if (in_arena) {
                    // a base cell outside b (the particle moved into a neighbour
                    // block) widens the group's stencils beyond the 6^3 nodes of b
                    if (ax0 == 0 || ax0 == 5 || ay0 == 0 || ay0 == 5 || az0 == 0 || az0 == 5) s.wide = 1u;
                    const int abase = ax0 + kAy * ay0 + kAz * az0;
                    const uint32_t cls = (uint32_t)abase & 31u;
                    s.st_key[slot] = (uint16_t)(cls | (atomicAdd(&s.ccount[cls], 1u) << 5));
                    s.st4[Smem::st(slot, 0)] = make_float4(ex, ey, ez, __int_as_float(abase));
                    s.st4[Smem::st(slot, 1)] = make_float4(qx, qy, qz, A[6]);
                    s.st4[Smem::st(slot, 2)] = make_float4(A[0], A[3], A[1], A[4]);
                    s.st4[Smem::st(slot, 3)] = make_float4(A[2], A[5], A[7], A[8]);
                    // bound of |q + A' o| over the stencil, per component: about its centre
                    // o = (1, 1, 1), or its base
                    auto bound_of = [](float q, float ai, float aj, float ak) {
                        const float r = fabsf(ai) + fabsf(aj) + fabsf(ak);
                        return USE == kStep ? fabsf(q + (ai + aj + ak)) + r : fabsf(q) + 2.f * r;
                    };
                    const float b0 = bound_of(qx, A[0], A[1], A[2]);
                    const float b1 = bound_of(qy, A[3], A[4], A[5]);
                    const float b2 = bound_of(qz, A[6], A[7], A[8]);
                    const float bp = fmaxf(fmaxf(b0, b1), b2);
                    bound = isfinite(bp) ? __float_as_uint(bp) : 0u;
                } else {
                    // moved further than one cell: scatter straight into G_{k+1}
                    s.st_key[slot] = Smem::kOut;
                    float wx2[3], wy2[3], wz2[3];
                    bspline_weights(ex, wx2);
                    bspline_weights(ey, wy2);
                    bspline_weights(ez, wz2);
                    for (int kk = 0; kk < 3; ++kk)
                        for (int jj = 0; jj < 3; ++jj) {
                            const float wjk = wy2[jj] * wz2[kk];
                            const float rx = qx + A[1] * jj + A[2] * kk;
                            const float ry = qy + A[4] * jj + A[5] * kk;
                            const float rz = qz + A[7] * jj + A[8] * kk;
                            for (int ii = 0; ii < 3; ++ii) {
                                const float w = wx2[ii] * wjk;
                                red_add4(&Gnext[node_addr_env(env, hx + ii, hy + jj, hz + kk, nb, nbe)],
                                         make_float4(w * m, w * (rx + A[0] * ii), w * (ry + A[3] * ii), w * (rz + A[6] * ii)));
                            }
                        }
                    for (int c = 0; c < 8; ++c) {
                        const int gi = (hx + 2 * (c & 1)) >> 2, gj = (hy + (c & 2)) >> 2, gk = (hz + ((c >> 1) & 2)) >> 2;
                        mark_clear(B, eb0 + block_id(gi, gj, gk, nb), step + 1, (step + 1u) % 3u);
                    }
                }
                // --- destination block of the new state
                int ddx = (hx >> 2) - bx, ddy = (hy >> 2) - by, ddz = (hz >> 2) - bz;
                if (ddx < -1 || ddx > 1 || ddy < -1 || ddy > 1 || ddz < -1 || ddz > 1) {
                    err |= kErrCfl;
                    ddx = min(max(ddx, -1), 1); ddy = min(max(ddy, -1), 1); ddz = min(max(ddz, -1), 1);
                }
                d = (ddx + 1) + 3 * (ddy + 1) + 9 * (ddz + 1);
            } else {
                s.st_key[slot] = Smem::kOut;
            }
            cp_async_commit();
            // --- stable rank by direction within the pass: per-warp counts, then
            // every warp derives the offsets it needs from the whole table (one
            // barrier per pass; warp 0 also publishes the pass's runs)
            uint32_t my_pos = (uint32_t)tid;              // position in the pass's output
            bool moved = valid && d != 13;                // to a neighbour block
            uint8_t(*wc)[Smem::NWP] = s.wcnt[pass & 1];
            unsigned peers = __ballot_sync(0xffffffffu, valid);
            if (__any_sync(0xffffffffu, moved)) peers = __match_any_sync(0xffffffffu, d);
            const uint32_t rank = __popc(peers & ((1u << lane) - 1u));
            if (valid && rank == 0) wc[d][warp] = (uint8_t)__popc(peers);
            bound = __reduce_max_sync(0xffffffffu, bound);
            if (lane == 0 && bound > 0u) atomicMax(&s.bmax, bound);
            // no particle of the pass left the block (most passes: a particle moves a
            // small part of a cell per sub-step): the order stays, one run
            moved = __syncthreads_or(moved);
            const uint32_t out_base = s.out_base, chunk_first = s.chunk_first;
            const uint32_t pbase = out_base + pass * T;
            const uint32_t npass_valid = min((uint32_t)T, total - pass * T);
            // lane l: the pass's particles in direction l (run), and those in directions
            // up to l (incl)
            uint32_t run = lane == 13 ? npass_valid : 0u, incl = npass_valid;
            if (moved) {
                uint32_t before = 0;                          // earlier warps' count of direction l
                run = 0;
                if (lane < 27) {
                    // byte sums by one multiply (four counts of at most 32: no carries)
                    auto bsum = [](uint32_t x) { return (x * 0x01010101u) >> 24; };
                    const uint32_t *cw = reinterpret_cast<const uint32_t *>(&wc[lane][0]);
                    uint32_t c[Smem::NWP / 4];
                    if (Smem::NWP == 16) *reinterpret_cast<uint4 *>(c) = *reinterpret_cast<const uint4 *>(cw);
                    else if (Smem::NWP == 8) *reinterpret_cast<uint2 *>(c) = *reinterpret_cast<const uint2 *>(cw);
                    else c[0] = cw[0];
#pragma unroll
                    for (int q = 0; q < Smem::NWP / 4; ++q) {
                        const int w = warp - 4 * q;      // earlier warps among this word's four
                        const uint32_t mk = w >= 4 ? 0xffffffffu : w <= 0 ? 0u : (1u << (8 * w)) - 1u;
                        run += bsum(c[q]);
                        before += bsum(c[q] & mk);
                    }
                }
                incl = run;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                my_pos = __shfl_sync(0xffffffffu, incl - run + before, d & 31) + rank;
            }
            // this warp's column of the other parity is next written by this warp, in
            // the next pass; every warp's reads of it ended before the barrier above
            if (lane < 28) s.wcnt[(pass + 1) & 1][lane][warp] = 0u;
            if (warp == 0 && chunk_first + pass < nchunk_cap) {
                if (lane < 27) {
                    B.chunks[0][chunk_out + chunk_first + pass].run[lane] = make_uint2(pbase + incl - run, run);
                    const int tx = bx + dir_dx(lane), ty = by + dir_dy(lane), tz = bz + dir_dz(lane);
                    if (run > 0u && tx >= 0 && ty >= 0 && tz >= 0 && tx < nb && ty < nb && tz < nb) {
                        uint4 *dst = (blk_out ? B.inbox[1] : B.inbox[0]) + (size_t)(eb0 + block_id(tx, ty, tz, nb)) * kInbox;
                        if (pass < (uint32_t)kNpMax)
                            dst[lane * kNpMax + pass] = make_uint4(pbase + incl - run, run, step + 1, 0u);
                        else
                            dst[kInbox - 1] = make_uint4(step + 1, 0u, 0u, 0u);   // overflow: use the run tables
                    }
                }
                const unsigned nz = __ballot_sync(0xffffffffu, lane < 27 && run > 0);
                if (lane == 0) s.mask |= nz;
            }
            const uint32_t pos = pbase + my_pos;
            if (RECORD && valid && pos < nparticles) {
                rec.xi[pos] = xi;
                rec.f0[pos] = a0;
                rec.f1[pos] = a1;
                rec.f2[pos] = f2;
                store_vc(rec.vc, pos, vx, vy, vz, Cm);
                rec.src[pos] = source_slot<MORE>(s, B, ncand, j);
            }
            if (valid && pos < nparticles) {
                B.P[0].xi[out_off + pos] = make_float4(nxp, nyp, nzp, idf);
                B.P[0].f0[out_off + pos] = make_float4(Fn[0], Fn[1], Fn[2], Fn[3]);
                B.P[0].f1[out_off + pos] = make_float4(Fn[4], Fn[5], Fn[6], Fn[7]);
                B.P[0].f2[out_off + pos] = Fn[8];
                if (WRITE_VC && last) store_vc(B.vc, pos, vx, vy, vz, Cm);
            }

            // --- P2G of the staged group (after every GP-th pass and the last one).
            // Lane l of warp w scatters staged slot 2 l + (w & 1) + 64 (w >> 1):
            // neighbouring lanes then hold particles of different cells.
            if (pass % GP == GP - 1 || pass + 1 == npass) {
                const int nstaged = (int)min((uint32_t)GROUP, total - (pass - pass % GP) * T);
                const float bmax = __uint_as_float(s.bmax);
                const bool wide = s.wide != 0u;
                const float sv = bmax > 0.f ? kFix / bmax : 1.0f;   // momentum fixed-point scale
                // order the group's arena particles by bank bucket (a counting sort over
                // 32 buckets): lane l of a warp then takes sorted position l * rows + j,
                // so the lanes of a warp sit in distinct banks at every stencil node
                const uint32_t cnt = s.ccount[lane];
                uint32_t cincl = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xffffffffu, cincl, o);
                    if (lane >= o) cincl += y;
                }
                const uint32_t nin = __shfl_sync(0xffffffffu, cincl, 31);
                const uint32_t cexcl = cincl - cnt;
#pragma unroll
                for (int p = 0; p < GP; ++p) {
                    const int sl = p * T + tid;
                    uint32_t key = sl < nstaged ? s.st_key[sl] : Smem::kOut;
                    const bool mine = key != Smem::kOut;
                    const uint32_t off = __shfl_sync(0xffffffffu, cexcl, key & 31u);
                    if (mine) s.order[off + (key >> 5)] = (uint16_t)sl;
                }
                __syncthreads();
                if (kEarly && pass + 1 == npass) mark_begin(s.mask);
                const uint32_t rows = (nin + 31u) >> 5;
                for (uint32_t jr = warp; jr < rows; jr += NW) {
                    const uint32_t pos = lane * rows + jr;
                    if (pos >= nin) continue;
                    const int q = s.order[pos];
                    const float4 c0 = s.st4[Smem::st(q, 0)], c1 = s.st4[Smem::st(q, 1)];
                    const float4 c2 = s.st4[Smem::st(q, 2)], c3 = s.st4[Smem::st(q, 3)];
                    const int base = __float_as_int(c0.w);
                    float wx[3], wy[3], wz[3];
                    bspline_weights(c0.x, wx);
                    bspline_weights(c0.y, wy);
                    bspline_weights(c0.z, wz);
                    // momentum inputs in fixed-point units, as (x, y) and (z, mass)
                    // pairs for the packed f32x2 pipe: the value at stencil offset
                    // (ii, jj, kk) is q + A' (ii, jj, kk), the mass term the constant
                    // kFix (m_p in mass units)
                    const float2 sv2 = make_float2(sv, sv), two = make_float2(2.f, 2.f);
                    const float2 qxy = __fmul2_rn(make_float2(c1.x, c1.y), sv2);
                    const float2 qzm = make_float2(c1.z * sv, kFix);
                    const float2 aixy = __fmul2_rn(make_float2(c2.x, c2.y), sv2);
                    const float2 ajxy = __fmul2_rn(make_float2(c2.z, c2.w), sv2);
                    const float2 akxy = __fmul2_rn(make_float2(c3.x, c3.y), sv2);
                    const float2 aizm = make_float2(c1.w * sv, 0.f);
                    const float2 ajzm = make_float2(c3.z * sv, 0.f);
                    const float2 akzm = make_float2(c3.w * sv, 0.f);
                    const float2 mm = make_float2(kMagic, kMagic);
                    const float2 wxx[3] = {make_float2(wx[0], wx[0]), make_float2(wx[1], wx[1]), make_float2(wx[2], wx[2])};
#pragma unroll
                    for (int kk = 0; kk < 3; ++kk) {
#pragma unroll
                        for (int jj = 0; jj < 3; ++jj) {
                            const float wjk = wy[jj] * wz[kk];
                            const float2 wjk2 = make_float2(wjk, wjk);
                            float2 rxy = qxy, rzm = qzm;
                            if (jj == 1) { rxy = __fadd2_rn(rxy, ajxy); rzm = __fadd2_rn(rzm, ajzm); }
                            if (jj == 2) { rxy = __ffma2_rn(two, ajxy, rxy); rzm = __ffma2_rn(two, ajzm, rzm); }
                            if (kk == 1) { rxy = __fadd2_rn(rxy, akxy); rzm = __fadd2_rn(rzm, akzm); }
                            if (kk == 2) { rxy = __ffma2_rn(two, akxy, rxy); rzm = __ffma2_rn(two, akzm, rzm); }
#pragma unroll
                            for (int ii = 0; ii < 3; ++ii) {
                                float2 vxy = rxy, vzm = rzm;
                                if (ii == 1) { vxy = __fadd2_rn(vxy, aixy); vzm = __fadd2_rn(vzm, aizm); }
                                if (ii == 2) { vxy = __ffma2_rn(two, aixy, vxy); vzm = __ffma2_rn(two, aizm, vzm); }
                                const float2 w2 = __fmul2_rn(wxx[ii], wjk2);
                                const float2 bxy = __ffma2_rn(w2, vxy, mm), bzm = __ffma2_rn(w2, vzm, mm);
                                const int a = base + ii + kAy * jj + kAz * kk;
                                atomicAdd(&s.acc[0][a], fix_round(bzm.y));
                                atomicAdd(&s.acc[1][a], fix_round(bxy.x));
                                atomicAdd(&s.acc[2][a], fix_round(bxy.y));
                                atomicAdd(&s.acc[3][a], fix_round(bzm.x));
                            }
                        }
                    }
                }
                __syncthreads();
                // arena -> G_{k+1}, then reset it for the next group: all 8^3 nodes,
                // or only the 6^3 around b when every base cell lies in b
                const float um = m / kFix, up = 1.0f / sv;
                const int nflush = wide ? 512 : 216;
                for (int q = tid; q < nflush; q += T) {
                    int lx8, ly8, lz8;
                    if (wide) {
                        lx8 = q & 7; ly8 = (q >> 3) & 7; lz8 = q >> 6;
                    } else {
                        lx8 = 1 + q % 6; ly8 = 1 + (q / 6) % 6; lz8 = 1 + q / 36;
                    }
                    const int a = lx8 + kAy * ly8 + kAz * lz8;
                    const int am = s.acc[0][a], px = s.acc[1][a], py = s.acc[2][a], pz = s.acc[3][a];
                    if (am != 0 || px != 0 || py != 0 || pz != 0) {
                        const int i = ox + lx8, jn = oy + ly8, k = oz + lz8;
                        if (i >= 0 && jn >= 0 && k >= 0 && i < n && jn < n && k < n)
                            red_add4(&Gnext[node_addr_env(env, i, jn, k, nb, nbe)],
                                     make_float4((float)am * um, (float)px * up, (float)py * up, (float)pz * up));
                        s.acc[0][a] = 0; s.acc[1][a] = 0; s.acc[2][a] = 0; s.acc[3][a] = 0;
                    }
                }
                if (kEarly && pass + 1 == npass) mark_end();
                // every thread read s.bmax, s.wide and the bucket sizes before the barriers
                // above; the next group's atomics come after the barrier below
                if (tid == 0) { s.bmax = 0; s.wide = 0; }
                if (tid < 32) s.ccount[tid] = 0u;
                __syncthreads();
            }
        }
        const uint32_t mask_b = s.mask;     // before warp 0 takes it for the next block
        cp_async_wait_all();
        __syncthreads();
        if (!kEarly || npass == 0) {
            mark_begin(mask_b);
            mark_end();
        }
    }

    if (err) atomicOr(&ctrl->err, err);
    const bool failed = __syncthreads_or(err != 0u);
    // Arrivals count up over the launch's sub-steps, target = CTAs x sub-steps so
    // far.  At the end of the launch's last one the last CTA reads part_alloc, whose
    // atomics every CTA consumed (its block's output range) before it arrived, and
    // the error bits, so that a CTA that set some releases them with a fence before
    // its arrival (the others need none); what the last CTA writes is read by the
    // next launch.  Elsewhere the arrival releases this CTA's writes and the wait
    // acquires the others'.
    if (last) {
        if (tid == 0) {
            if (failed) __threadfence();
            if (atomicAdd(&ctrl->done, 1u) == target - 1u) {
                __threadfence();
                // one round trip for all three; an append to the next sub-step's list that is
                // not ordered before its CTA's arrival may be missing from it (the host only
                // weighs configurations by the blocks)
                const uint32_t handed_out = *(volatile uint32_t *)&ctrl->part_alloc[m3];
                uint32_t bits = *(volatile uint32_t *)&ctrl->err;
                unsigned long long next = 0;
                if constexpr (kGated<MINB, USE>)
                    next = *(volatile unsigned long long *)&ctrl->nactive[s.m3 == 2u ? 0u : s.m3 + 1u][0];
                if (handed_out != nparticles) {
                    bits |= kErrCapacity;
                    atomicOr(&ctrl->err, kErrCapacity);
                }
                ctrl->done = 0;
                *(volatile uint32_t *)B.host_err = bits;
                if constexpr (kGated<MINB, USE>)
                    *(volatile unsigned long long *)B.host_blocks =
                        (unsigned long long)((uint32_t)next + (uint32_t)(next >> 32)) << 32 | (step + 1u);
                ctrl->step = step + 1;
            }
        }
        return false;
    }
    if (tid == 0) {
        // every CTA is resident (cooperative launch), so the wait ends when the last
        // one arrives; after max_polls looks it ends with an error.  A CTA whose own
        // look comes after the last arrival still goes on: every arrival was made, so it
        // finds the sub-step before complete, and leaves at the next wait.
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&ctrl->done) : "memory");
        uint32_t now, polls = 0;
        do {
            asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(now) : "l"(&ctrl->done) : "memory");
        } while (now < target && ++polls < B.max_polls);
        asm volatile("fence.acq_rel.gpu;" ::: "memory");
        if (now < target) {    // nobody reaches the end of the launch, where step and the host's copy are written
            *(volatile uint32_t *)&ctrl->step = kStepStalled;
            *(volatile uint32_t *)B.host_err = atomicOr(&ctrl->err, kErrStall) | kErrStall;
        }
        s.go = now >= target;
    }
    __syncthreads();
    return s.go;
}

// Launches of several sub-steps where the registers allow it.  A small scene's
// sub-step is one block's chain of round trips plus the launch gap and the ramp
// of its CTAs; without the latter two, and with the neighbour marks begun before
// the last scatter, the 30K slab takes 13.8 instead of 16.5 us per sub-step of a
// 25-sub-step frame (256 threads, 2 CTAs per SM) and the 8K cube 22.4 -> 21.8.  At 80
// registers a thread the loop's state spills: 1M particles 94.6 -> 106 us.
template <int T, int MINB>
constexpr bool kManySteps = T * MINB <= 640;

// nsub sub-steps, the tool frames of each `frames` entries after the one
// before.  One launch for all of them spares the launch gap and the ramp of the
// CTAs between sub-steps; the CTAs then wait for one another, so nsub > 1 needs
// a cooperative launch.  v and C are written by the last one (if WRITE_VC).
template <bool WRITE_VC, int T, int GP, int MINB = kMinBlocks<T, GP>, Use USE = kStep, int PD = 1, bool MORE = false>
__global__ void __launch_bounds__(T, MINB) k_fused_step(DevParams P, FusedBufs B,
                                                        const ToolFrame *__restrict__ tools, uint32_t frames,
                                                        StepRecord rec, uint32_t nsub, LaunchGate gate) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FusedSmem<T, GP, PD> &s = *reinterpret_cast<FusedSmem<T, GP, PD> *>(smem_raw);
    const uint32_t step = *(volatile uint32_t *)&B.ctrl->step;
    // Behind a wait that ran out, the arrivals, counters and lists are those of a launch
    // that its CTAs left at different sub-steps: nothing runs on them before the next
    // load sets them anew.  (That keeps the lists in bounds: a block is appended once
    // per stamp, to a counter that was zero.)
    if (step == kStepStalled) return;
    if constexpr (kGated<MINB, USE>) {
        if (gate.at != LaunchGate::kAny && step != gate.at) return;
        if (gate.most_blocks != LaunchGate::kAny) {
            const unsigned long long nhl = *(volatile unsigned long long *)&B.ctrl->nactive[step % 3u][0];
            if ((uint32_t)nhl + (uint32_t)(nhl >> 32) > gate.most_blocks) return;
        }
    }
    if constexpr (!kManySteps<T, MINB>) {
        fused_substep<WRITE_VC, T, GP, MINB, USE, PD, MORE>(s, P, B, tools, rec, 0, step, gridDim.x, true, true);
    } else {
        for (uint32_t k = 0;; ++k)
            if (!fused_substep<WRITE_VC, T, GP, MINB, USE, PD, MORE>(s, P, B, tools + (size_t)k * frames, rec, k, step + k,
                                                                  (k + 1) * gridDim.x, k == 0, k + 1 == nsub))
                break;
    }
}

// nsub sub-steps as one launch, cooperative if there are several, or one by one
// where the CTAs cannot all be resident (a context with a part of the SMs).
template <typename Kernel>
void launch_steps(Kernel kernel, int threads, size_t smem, const DevParams &P, const FusedBufs &B, const ToolFrame *tools,
                  const StepRecord &rec, int nsub, int grid, cudaStream_t st, const LaunchGate &gate = {}) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = threads;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = nsub > 1 ? 1 : 0;
    const uint32_t frames = (uint32_t)(P.n_envs * P.tstride);
    // a failure is left for cudaGetLastError
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, P, B, tools, frames, rec, (uint32_t)nsub, gate);
    if (nsub > 1 && (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported)) {
        cudaGetLastError();
        cfg.numAttrs = 0;
        for (int k = 0; k < nsub; ++k) {
            LaunchGate g = gate;       // decided for the first sub-step; the others follow it
            if (k > 0 && g.at != LaunchGate::kAny) {
                g.at += (uint32_t)k;
                g.most_blocks = LaunchGate::kAny;
            }
            cudaLaunchKernelEx(&cfg, kernel, P, B, tools + (size_t)k * frames, frames, record_of(rec, k), 1u, g);
        }
    }
}

// The kernel of a configuration, as FusedBufs::runs is there or not.
template <bool WRITE_VC, int T, int GP, int MINB, int PD>
auto step_kernel(bool more) {
    if constexpr (T < 256)
        if (more) return k_fused_step<WRITE_VC, T, GP, MINB, kStep, PD, true>;
    return k_fused_step<WRITE_VC, T, GP, MINB, kStep, PD>;
}

// With 128 registers the variant that writes v and C does not spill either, and
// all sub-steps are one launch; otherwise the last is its own.
template <int T, int GP, int MINB = kMinBlocks<T, GP>, int PD = 1>
void launch_variant(const DevParams &P, const FusedBufs &B, const ToolFrame *tools, int nsub, bool write_vc, int grid,
                    cudaStream_t st, const LaunchGate &gate = {}) {
    constexpr bool kOne = T * MINB <= 512;
    const size_t smem = sizeof(FusedSmem<T, GP, PD>), frames = (size_t)P.n_envs * P.tstride;
    const StepRecord none{};
    const int plain = !write_vc ? nsub : kOne ? 0 : nsub - 1;
    const int per = kManySteps<T, MINB> ? plain : 1;
    for (int k = 0; k < plain; k += per)
        launch_steps(step_kernel<false, T, GP, MINB, PD>(B.runs != nullptr), T, smem, P, B, tools + k * frames, none, per, grid, st,
                     gate);
    if (plain < nsub)
        launch_steps(step_kernel<true, T, GP, MINB, PD>(B.runs != nullptr), T, smem, P, B, tools + plain * frames, none,
                     nsub - plain, grid, st, gate);
}

template <int T, int GP, int MINB = kMinBlocks<T, GP>, int PD = 1>
int variant_occupancy(bool more) {
    const int bytes = (int)sizeof(FusedSmem<T, GP, PD>);
    int least = INT_MAX;
    for (const auto kernel : {step_kernel<true, T, GP, MINB, PD>(more), step_kernel<false, T, GP, MINB, PD>(more)}) {
        int ctas = 0;
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ctas, kernel, T, bytes);
        least = std::min(least, ctas);
    }
    return least;
}

}  // namespace

void launch_fused_steps(const DevParams &P, const FusedBufs &B, const ToolFrame *tools, int nsub, bool write_vc,
                        int grid, int config, cudaStream_t st, const LaunchGate &gate) {
    switch (config) {
    case 1: launch_variant<256, 1>(P, B, tools, nsub, write_vc, grid, st); break;
    case 2: launch_variant<128, 2, kMinBlocks<128, 2>, 2>(P, B, tools, nsub, write_vc, grid, st); break;
    case 3: launch_variant<128, 1>(P, B, tools, nsub, write_vc, grid, st); break;
    case 4: launch_variant<256, 2, 2, 2>(P, B, tools, nsub, write_vc, grid, st, gate); break;   // 2 CTAs per SM, 128 registers
    case 5: launch_variant<512, 2>(P, B, tools, nsub, write_vc, grid, st, gate); break;         // 1 CTA per SM, 128 registers
    default: launch_variant<256, 2>(P, B, tools, nsub, write_vc, grid, st); break;
    }
}

bool fused_many_steps(int config) { return config != 0 && config != 1; }

int fused_step_threads(int config) { return config == 5 ? 512 : config == 2 || config == 3 ? 128 : 256; }

// The sub-steps of a recorded rollout: 256 threads, 2 passes per flush and 2
// CTAs per SM (128 registers); the recording ones copy particles one pass ahead.
int fused_rollout_occupancy() {
    constexpr int rec = (int)sizeof(FusedSmem<256, 2>), fwd = (int)sizeof(FusedSmem<256, 2, 2>);
    cudaFuncSetAttribute(k_fused_step<false, 256, 2, 2, kRecord>, cudaFuncAttributeMaxDynamicSharedMemorySize, rec);
    cudaFuncSetAttribute(k_fused_step<true, 256, 2, 2, kRollout, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, fwd);
    int a = 0, b = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_fused_step<false, 256, 2, 2, kRecord>, 256, rec);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_fused_step<true, 256, 2, 2, kRollout, 2>, 256, fwd);
    return a < b ? a : b;
}

void launch_fused_step_record(const DevParams &P, const FusedBufs &B, const ToolFrame *tools, const StepRecord &rec,
                              int nsub, int grid, cudaStream_t st) {
    launch_steps(k_fused_step<false, 256, 2, 2, kRecord>, 256, sizeof(FusedSmem<256, 2>), P, B, tools, rec, nsub, grid,
                 st);
}

void launch_fused_steps_rollout(const DevParams &P, const FusedBufs &B, const ToolFrame *tools, int nsub, int grid,
                                cudaStream_t st) {
    launch_steps(k_fused_step<true, 256, 2, 2, kRollout, 2>, 256, sizeof(FusedSmem<256, 2, 2>), P, B, tools,
                 StepRecord{}, nsub, grid, st);
}

// Also opts the kernel into its dynamic shared memory size on the current
// device; called when a handle is created.
int fused_step_occupancy(int config, bool more) {
    switch (config) {
    case 1: return variant_occupancy<256, 1>(more);
    case 2: return variant_occupancy<128, 2, kMinBlocks<128, 2>, 2>(more);
    case 3: return variant_occupancy<128, 1>(more);
    case 4: return variant_occupancy<256, 2, 2, 2>(more);
    case 5: return variant_occupancy<512, 2>(more);
    default: return variant_occupancy<256, 2>(more);
    }
}

}  // namespace gbmpm
