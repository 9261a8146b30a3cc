// kernels_surface.cu -- iso-surface extraction of the grid density, the
// renderer's Marching Cubes step (Sec. III), in its tetrahedral form: every
// cell is split into six tetrahedra around its diagonal from corner 0 to
// corner 7 (corner c at offset (c & 1, (c >> 1) & 1, (c >> 2) & 1)), each of
// which contributes 0, 1 or 2 triangles facing away from the inside
// (density >= iso).  Neighbouring cells split their shared faces alike, so
// the surface is closed.  Triangles are written in cell order (i fastest).
//
// The grid is read once, for one inside bit per node (2 MB per 256^3 nodes
// against 268 MB of grid); counting works on words of 32 cells of a row, bit
// by bit in parallel, and the emitting warps touch the density only at the
// edges of the triangles they write, one lane per vertex, so that a warp's
// stores are contiguous.  A cell's triangles come from a table over its eight
// inside bits, built by the compiler.
// 300K-particle slab on the 128^3 grid, per-cell counts and scans over all 2M
// cells and a triangle loop per cell before: 103 -> 54 us a call.
#include "common.cuh"
#include "launch.h"

namespace gbmpm {

namespace {

constexpr int kScanBlock = 1024;
constexpr int kUnit = 32;             // words of cells per prefix entry
constexpr int kParts = 8;             // emitting warps per unit, each the words of one remainder mod kParts:
                                      // the words of a row lie in different warps
constexpr int kEmitWarps = 8;         // warps per emitting CTA

// Per corner mask (bit c: corner c inside) the cell's triangles, tetrahedron by
// tetrahedron: three edges of two corners (3 bits each, the lower-numbered one
// first), and their number.
struct SurfaceTable {
    alignas(16) uint32_t tri[256][12];
    uint8_t count[256];
};

// The six tetrahedra (0, a, b, 7) along the paths 0 -> a -> b -> 7, with
// corners 1 and 2 swapped where needed for a positive orientation (sign of
// det[B - A, C - A, D - A] over the integer corner offsets).
constexpr void tetrahedron(int q, int t[4]) {
    const int pa[6] = {1, 1, 2, 2, 4, 4}, pb[6] = {3, 5, 3, 6, 5, 6};
    t[0] = 0; t[1] = pa[q]; t[2] = pb[q]; t[3] = 7;
    int u[3] = {}, v[3] = {}, w[3] = {};
    for (int a = 0; a < 3; ++a) {
        u[a] = (t[1] >> a) & 1;
        v[a] = (t[2] >> a) & 1;
        w[a] = (t[3] >> a) & 1;
    }
    const int det = u[0] * (v[1] * w[2] - v[2] * w[1]) - u[1] * (v[0] * w[2] - v[2] * w[0]) +
                    u[2] * (v[0] * w[1] - v[1] * w[0]);
    if (det < 0) { const int x = t[1]; t[1] = t[2]; t[2] = x; }
}

constexpr uint32_t edge_code(int a, int b) { return a < b ? (uint32_t)(a | b << 3) : (uint32_t)(b | a << 3); }
constexpr uint32_t tri_code(uint32_t e0, uint32_t e1, uint32_t e2) { return e0 | e1 << 6 | e2 << 12; }

constexpr SurfaceTable make_surface_table() {
    SurfaceTable T = {};
    for (int code = 0; code < 256; ++code) {
        int cnt = 0;
        for (int q = 0; q < 6; ++q) {
            int t[4] = {};
            tetrahedron(q, t);
            int in[4] = {}, nin = 0;
            for (int r = 0; r < 4; ++r) { in[r] = (code >> t[r]) & 1; nin += in[r]; }
            if (nin == 1 || nin == 3) {
                // the lone vertex first, in an even permutation of t
                int lone = 0;
                for (int r = 0; r < 4; ++r) if (in[r] == (nin == 1)) lone = r;
                const int perms[4][4] = {{0, 1, 2, 3}, {1, 0, 3, 2}, {2, 0, 1, 3}, {3, 0, 2, 1}};
                const int *p = perms[lone];
                const uint32_t e0 = edge_code(t[p[0]], t[p[1]]), e1 = edge_code(t[p[0]], t[p[2]]),
                               e2 = edge_code(t[p[0]], t[p[3]]);
                // three inside: the inside is on the other side, so reversed
                T.tri[code][cnt++] = nin == 1 ? tri_code(e0, e1, e2) : tri_code(e0, e2, e1);
            } else if (nin == 2) {
                // inside (p, q), outside (r, s) in an even permutation of t: the
                // quad pr, ps, qs, qr as two triangles
                int perm[4] = {}, a = 0, b = 2;
                for (int r = 0; r < 4; ++r) { if (in[r]) perm[a++] = r; else perm[b++] = r; }
                int inv = 0;
                for (int x = 0; x < 4; ++x)
                    for (int y = x + 1; y < 4; ++y) inv += perm[x] > perm[y];
                if (inv & 1) { const int x = perm[2]; perm[2] = perm[3]; perm[3] = x; }
                const int P = t[perm[0]], Q = t[perm[1]], R = t[perm[2]], S = t[perm[3]];
                T.tri[code][cnt++] = tri_code(edge_code(P, R), edge_code(P, S), edge_code(Q, S));
                T.tri[code][cnt++] = tri_code(edge_code(P, R), edge_code(Q, S), edge_code(Q, R));
            }
        }
        T.count[code] = (uint8_t)cnt;
    }
    return T;
}
__device__ constexpr SurfaceTable d_table = make_surface_table();

// Inside bits: bit i & 31 of word (k n + j) W + i / 32, W = ceil(n / 32).  A
// warp takes one word of the four rows of a grid block, whose 64-byte pieces
// share 128-byte lines.
__global__ void __launch_bounds__(256) k_surface_bits(const float4 *__restrict__ G, int n, int nb, uint32_t nbe,
                                                       uint32_t env, float scale, float iso, uint32_t *__restrict__ bits) {
    const uint32_t W = (uint32_t)(n + 31) / 32u, lane = threadIdx.x & 31u;
    const uint32_t items = (uint32_t)n * (uint32_t)nb * W, stride = gridDim.x * (blockDim.x >> 5);
    for (uint32_t it = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); it < items; it += stride) {
        const uint32_t w = it % W, jb = it / W % (uint32_t)nb, k = it / (W * (uint32_t)nb);
        const int i = (int)(32u * w + lane);
        bool in[4];
#pragma unroll
        for (int r = 0; r < 4; ++r)
            in[r] = i < n && __fmul_rn(__ldg(&G[node_addr_env(env, i, (int)(4 * jb) + r, (int)k, nb, nbe)].x), scale) >= iso;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const uint32_t m = __ballot_sync(0xffffffffu, in[r]);
            if (lane == 0) bits[(k * (uint32_t)n + 4 * jb + r) * W + w] = m;
        }
    }
}

// The eight corner words of cell word g (32 cells of row (j, k), j, k < n - 1)
// and the cells of it that exist.
__device__ __forceinline__ uint32_t corner_words(const uint32_t *__restrict__ bits, uint32_t g, int n, uint32_t W,
                                                 uint32_t c[8], uint32_t &w, uint32_t &j, uint32_t &k) {
    const uint32_t m = (uint32_t)n - 1u;
    w = g % W; j = g / W % m; k = g / (W * m);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const uint32_t *row = bits + ((k + (r >> 1)) * (uint32_t)n + j + (r & 1)) * W + w;
        const uint32_t lo = __ldg(row), hi = w + 1u < W ? __ldg(row + 1) : 0u;
        c[2 * r] = lo;
        c[2 * r + 1] = __funnelshift_r(lo, hi, 1);
    }
    const uint32_t left = m - 32u * w;      // cells from this word's first one on
    return left >= 32u ? 0xffffffffu : (1u << left) - 1u;
}

// Triangles per word of cells, and their sum per kUnit words.  A tetrahedron
// with one or three corners inside (odd parity) gives one, with two gives two.
__global__ void __launch_bounds__(256) k_surface_count(const uint32_t *__restrict__ bits, int n,
                                                        uint16_t *__restrict__ counts, uint32_t *__restrict__ sums) {
    const uint32_t W = (uint32_t)(n + 31) / 32u, m = (uint32_t)n - 1u, words = m * m * W;
    const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    uint32_t cnt = 0;
    if (g < words) {
        uint32_t c[8], w, j, k;
        const uint32_t valid = corner_words(bits, g, n, W, c, w, j, k);
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            // corners along the path 0 -> a -> b -> 7
            const int pa[6] = {1, 1, 2, 2, 4, 4}, pb[6] = {3, 5, 3, 6, 5, 6};
            const uint32_t a = c[0], b = c[pa[q]], d = c[pb[q]], e = c[7];
            const uint32_t odd = a ^ b ^ d ^ e;
            const uint32_t mixed = (a | b | d | e) & ~(a & b & d & e);
            cnt += __popc(odd & valid) + 2 * __popc(mixed & ~odd & valid);
        }
        counts[g] = (uint16_t)cnt;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    if ((threadIdx.x & 31) == 0 && g < words) sums[g / kUnit] = cnt;
}

// exclusive scan over a CTA
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t *s_warp, uint32_t &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < (int)(blockDim.x >> 5) ? s_warp[lane] : 0u;
        uint32_t wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += y;
        }
        s_warp[lane] = wi - w;
        if (lane == 31) s_warp[32] = wi;
    }
    __syncthreads();
    total = s_warp[32];
    const uint32_t r = s_warp[warp] + incl - v;
    __syncthreads();
    return r;
}

// one CTA: exclusive scan of the unit sums, and the grand total at sums[nblk]
__global__ void __launch_bounds__(kScanBlock) k_scan_sums(uint32_t *__restrict__ sums, uint32_t nblk) {
    __shared__ uint32_t s_warp[33];
    uint32_t carry = 0;
    for (uint32_t base = 0; base < nblk; base += kScanBlock) {
        const uint32_t i = base + threadIdx.x;
        const uint32_t v = i < nblk ? sums[i] : 0u;
        uint32_t total;
        const uint32_t e = block_exclusive_scan(v, s_warp, total);
        if (i < nblk) sums[i] = carry + e;
        carry += total;
    }
    if (threadIdx.x == 0) sums[nblk] = carry;
}

__device__ __forceinline__ uint32_t warp_exclusive_scan(uint32_t v, int lane) {
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    return incl - v;
}

// Triangles of a unit's words of cells, a part of them per warp, one vertex per
// lane: the point where the density crosses iso on an edge, computed from its
// lower-numbered corner.  A lane first brings the corner densities of its own
// cell into shared memory, so that a word costs two round trips, not one per
// vertex.
__global__ void __launch_bounds__(32 * kEmitWarps) k_surface_emit(const float4 *__restrict__ G, int n, int nb,
                                                                  uint32_t nbe, uint32_t env, float scale, float iso,
                                                                  float dx, const uint32_t *__restrict__ bits,
                                                                  const uint16_t *__restrict__ counts,
                                                                  const uint32_t *__restrict__ sums,
                                                                  float *__restrict__ tri, uint64_t max_tri) {
    __shared__ uint32_t s_list[kEmitWarps][32 * 12];     // a word's triangles: cell (5 bits), table entry
    __shared__ float s_f[kEmitWarps][32 * 9];            // and its cells' corner densities, 9 apart
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t W = (uint32_t)(n + 31) / 32u, m = (uint32_t)n - 1u, words = m * m * W;
    const uint32_t part = (blockIdx.x * kEmitWarps + warp) % kParts, u = (blockIdx.x * kEmitWarps + warp) / kParts;
    if (u * kUnit >= words) return;
    const uint32_t first = sums[u];
    if (sums[u + 1] == first || first >= max_tri) return;
    const uint32_t cnt_w = u * kUnit + lane < words ? counts[u * kUnit + lane] : 0u;
    const uint32_t off_w = first + warp_exclusive_scan(cnt_w, lane);
    uint32_t *list = s_list[warp];
    float *fc = s_f[warp];
    uint32_t todo = __ballot_sync(0xffffffffu, cnt_w > 0u && lane % kParts == part);
    for (; todo; todo &= todo - 1u) {
        const int wl = __ffs(todo) - 1;
        const uint32_t total = __shfl_sync(0xffffffffu, cnt_w, wl), base = __shfl_sync(0xffffffffu, off_w, wl);
        uint32_t c[8], w, j, k;
        const uint32_t valid = corner_words(bits, u * kUnit + wl, n, W, c, w, j, k);
        uint32_t code = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) code |= ((c[q] >> lane) & 1u) << q;
        const uint32_t cnt = (valid >> lane) & 1u ? d_table.count[code] : 0u;
        const uint32_t pos = warp_exclusive_scan(cnt, lane);
        __syncwarp();
        if (cnt > 0u) {
#pragma unroll
            for (int q = 0; q < 8; ++q)      // rounded before its use, as the inside bits are
                fc[9 * lane + q] =
                    __fmul_rn(__ldg(&G[node_addr_env(env, (int)(32u * w) + lane + (q & 1), (int)j + ((q >> 1) & 1),
                                                     (int)k + (q >> 2), nb, nbe)].x), scale);
        }
        if (cnt > 0u) {
            const uint4 *row = reinterpret_cast<const uint4 *>(d_table.tri[code]);
            const uint4 e0 = row[0], e1 = row[1], e2 = row[2];
            const uint32_t e[12] = {e0.x, e0.y, e0.z, e0.w, e1.x, e1.y, e1.z, e1.w, e2.x, e2.y, e2.z, e2.w};
#pragma unroll
            for (uint32_t t = 0; t < 12u; ++t)
                if (t < cnt) list[pos + t] = e[t] << 5 | (uint32_t)lane;
        }
        __syncwarp();
        for (uint32_t v = lane; v < 3 * total; v += 32) {
            const uint32_t t = v / 3u, e = list[t];
            const uint32_t edge = e >> (5u + 6u * (v - 3u * t));
            const int a = edge & 7u, b = (edge >> 3) & 7u;
            const int cell = (int)(e & 31u), i = (int)(32u * w) + cell;
            const float fa = fc[9 * cell + a], fb = fc[9 * cell + b];
            const int ai = i + (a & 1), aj = (int)j + ((a >> 1) & 1), ak = (int)k + (a >> 2);
            const float s = (iso - fa) / (fb - fa);
            if ((uint64_t)base + t < max_tri) {
                float *out = tri + 9 * ((size_t)base + t) + 3 * (v - 3u * t);
                out[0] = ((float)ai + s * (float)((b & 1) - (a & 1))) * dx;
                out[1] = ((float)aj + s * (float)(((b >> 1) & 1) - ((a >> 1) & 1))) * dx;
                out[2] = ((float)ak + s * (float)((b >> 2) - (a >> 2))) * dx;
            }
        }
    }
}

}  // namespace

SurfaceSizes surface_sizes(int n) {
    const size_t W = (size_t)(n + 31) / 32, m = (size_t)n - 1;
    SurfaceSizes z;
    z.bits = (size_t)n * n * W;
    z.words = m * m * W;
    z.units = (z.words + kUnit - 1) / kUnit;
    return z;
}

void launch_surface_count(const float4 *G, int n, int nb, uint32_t nbe, uint32_t env, float scale, float iso,
                          const SurfaceScratch &S, int grid, cudaStream_t st) {
    const SurfaceSizes z = surface_sizes(n);
    k_surface_bits<<<grid, 256, 0, st>>>(G, n, nb, nbe, env, scale, iso, S.bits);
    k_surface_count<<<(unsigned)((z.words + 255) / 256), 256, 0, st>>>(S.bits, n, S.counts, S.sums);
    k_scan_sums<<<1, kScanBlock, 0, st>>>(S.sums, (uint32_t)z.units);
}

void launch_surface_emit(const float4 *G, int n, int nb, uint32_t nbe, uint32_t env, float scale, float iso, float dx,
                         const SurfaceScratch &S, float *tri, uint64_t max_tri, cudaStream_t st) {
    const size_t warps = surface_sizes(n).units * kParts;
    k_surface_emit<<<(unsigned)((warps + kEmitWarps - 1) / kEmitWarps), 32 * kEmitWarps, 0, st>>>(
        G, n, nb, nbe, env, scale, iso, dx, S.bits, S.counts, S.sums, tri, max_tri);
}

}  // namespace gbmpm
