// Voxel radiance cache (Sec. 4.2): the input pixels' radiance is
// average-pooled onto an R^3 grid spanned over the scene box and queried at
// the voxel containing a hit point (the paper uses R = 256).  Pixels are
// assigned to voxels as correctly rounded FP64 operations place them (as
// the Morton quantisation), grouped by a stable radix sort on the voxel
// index, and each voxel's mean is its FP64 sum in pixel order over the
// count, so the grid is deterministic.  GB300 runs FP64 at 1/64 of the
// float32 rate, so both steps reach those FP64 results by cheaper exact
// means: cells in float32 away from cell faces, sums in integers while
// they are provably exact (k_vox_keys, k_vox_means), FP64 otherwise.
#include "fipt_internal.cuh"
#include "exact_sum.cuh"

namespace {

// The per-axis scale R / (hi - lo) is the same correctly rounded double for
// every pixel; the first three threads of a block compute it once.
//
// A pixel's cell on an axis is floor(RN64(RN64(x - lo) * scale)), clamped
// to [0, R - 1].  Most cells are found in float32 without changing that
// result: f = RN32(RN32(x - lo) * RN32(scale)) and the FP64 value both lie
// within relative 2^-24 (three roundings) plus 2^-53 (two) of the exact
// product, so |f - f64| < 2^-22 |f| away from underflow.  When no integer
// in [1, R - 1] lies within 2^-21 |f| of f, no cell face separates f from
// the FP64 value and floor(f) clamps to the same cell; a cell face at 0 or
// R clamps either side to the same cell, and an f that underflows keeps
// the sign of x - lo.  Pixels near an inner cell face (and NaNs) take the
// FP64 arithmetic, and so does every pixel on an axis whose float32 scale
// is infinite or subnormal (extents below ~1e-35 or near 1e38), where the
// bound does not hold.
__global__ void k_vox_keys(const float* __restrict__ x, int64_t stride, int64_t P,
                           const SceneConst* __restrict__ c, int R, uint32_t* __restrict__ keys,
                           uint32_t* __restrict__ vals) {
    __shared__ double scale[3];
    __shared__ float scale32[3];
    __shared__ bool fast[3];
    if (threadIdx.x < 3) {
        const double ext = __dsub_rn((double)c->hi[threadIdx.x], (double)c->lo[threadIdx.x]);
        scale[threadIdx.x] = ext > 0.0 ? __ddiv_rn((double)R, ext) : 0.0;
        const float s32 = __double2float_rn(scale[threadIdx.x]);
        scale32[threadIdx.x] = s32;
        fast[threadIdx.x] = s32 == 0.0f || (s32 >= 1.17549435e-38f && s32 <= 3.40282347e38f);
    }
    __syncthreads();
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= P) return;
    uint32_t ix[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float xa = x[p * stride + a];
        const float lo32 = c->lo[a];
        const float f = __fmul_rn(__fsub_rn(xa, lo32), scale32[a]);
        const float r = rintf(f);
        const bool near_face = r >= 1.0f && r <= (float)(R - 1) && fabsf(f - r) <= fabsf(f) * 0x1p-21f;
        if (fast[a] && !near_face && f == f) {
            const float fl = floorf(f);
            ix[a] = fl < 0.0f ? 0u : (fl > (float)(R - 1) ? (uint32_t)(R - 1) : (uint32_t)fl);
        } else {
            const double lo = (double)lo32;
            double g = 0.0;
            if (scale[a] > 0.0) g = __dmul_rn(__dsub_rn((double)xa, lo), scale[a]);
            double fl = floor(g);
            fl = fl < 0.0 ? 0.0 : (fl > (double)(R - 1) ? (double)(R - 1) : fl);
            ix[a] = (uint32_t)fl;
        }
    }
    keys[p] = (ix[2] * (uint32_t)R + ix[1]) * (uint32_t)R + ix[0];
    vals[p] = (uint32_t)p;
}

// Run heads (the first sorted pixel of each voxel's run) listed in pixel
// order, so that run h spans [heads[h], heads[h + 1]) with heads[nh] = P:
// k_vox_count counts the heads of each tile of HEAD_TILE pixels,
// k_vox_scan turns the counts into offsets (one block) and k_vox_compact
// writes each tile's heads at its offset.
constexpr int HEAD_TILE = 1024;

__device__ __forceinline__ bool run_head(const uint32_t* __restrict__ keys, int64_t j, int64_t P) {
    return j < P && (j == 0 || keys[j - 1] != keys[j]);
}

// Exclusive prefix of v over the block's 32 warps (v given by lane 0 of
// each warp in ws[w]); ws[w] becomes the sum of warps before w and the
// return value (all threads) the block total.
__device__ __forceinline__ uint32_t warp_offsets(uint32_t* ws) {
    __syncthreads();
    const int lane = threadIdx.x & 31;
    if (threadIdx.x < 32) {
        const uint32_t v = ws[lane];
        uint32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        ws[lane] = x - v;
        if (lane == 31) ws[32] = x;
    }
    __syncthreads();
    return ws[32];
}

__global__ void __launch_bounds__(HEAD_TILE)
k_vox_count(const uint32_t* __restrict__ keys, int64_t P, uint32_t* __restrict__ tcount) {
    __shared__ uint32_t ws[33];
    const int64_t j = blockIdx.x * (int64_t)HEAD_TILE + threadIdx.x;
    const unsigned m = __ballot_sync(0xffffffffu, run_head(keys, j, P));
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = __popc(m);
    const uint32_t total = warp_offsets(ws);
    if (threadIdx.x == 0) tcount[blockIdx.x] = total;
}

// One block: exclusive scan of the nt tile counts in place, nh = their sum,
// heads[nh] = P.
__global__ void __launch_bounds__(HEAD_TILE)
k_vox_scan(uint32_t* __restrict__ tcount, int64_t nt, uint32_t* __restrict__ heads, uint32_t* __restrict__ nhead,
           int64_t P) {
    __shared__ uint32_t ws[33];
    const int lane = threadIdx.x & 31;
    uint32_t carry = 0;
    for (int64_t base = 0; base < nt; base += HEAD_TILE) {
        const int64_t i = base + threadIdx.x;
        const uint32_t v = i < nt ? tcount[i] : 0u;
        uint32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) ws[threadIdx.x >> 5] = x;
        const uint32_t total = warp_offsets(ws);
        if (i < nt) tcount[i] = carry + ws[threadIdx.x >> 5] + x - v;
        carry += total;
        __syncthreads();                         // ws is rewritten by the next chunk
    }
    if (threadIdx.x == 0) {
        *nhead = carry;
        heads[carry] = (uint32_t)P;
    }
}

__global__ void __launch_bounds__(HEAD_TILE)
k_vox_compact(const uint32_t* __restrict__ keys, int64_t P, const uint32_t* __restrict__ toff,
              uint32_t* __restrict__ heads) {
    __shared__ uint32_t ws[33];
    const int lane = threadIdx.x & 31;
    const int64_t j = blockIdx.x * (int64_t)HEAD_TILE + threadIdx.x;
    const bool h = run_head(keys, j, P);
    const unsigned m = __ballot_sync(0xffffffffu, h);
    if (lane == 0) ws[threadIdx.x >> 5] = __popc(m);
    warp_offsets(ws);
    if (h) heads[toff[blockIdx.x] + ws[threadIdx.x >> 5] + __popc(m & ((1u << lane) - 1u))] = (uint32_t)j;
}

constexpr int MEAN_THREADS = 128;
constexpr int MEAN_LANES = 8;    // lanes per run where the runs are long
constexpr int MEAN_UNIT = MEAN_THREADS / MEAN_LANES;     // runs of a block there
constexpr int MEAN_SUBS = MEAN_THREADS / MEAN_UNIT;      // and such blocks per run of each thread
constexpr int MEAN_SHORT = 4;    // pixels per run, over MEAN_THREADS neighbouring runs, up to which they are short
constexpr int VU = 4;            // pixels a lane takes at a time

// The sums of one run per LANES lanes (lane c of them, run [j0, j1) of count
// pixels, the same for all), which take its pixels LANES * VU at a time, the next
// pixel indices loading while this group's radiance is fetched.  Each channel's
// FP64 sum in pixel order is carried exactly in integers (exact_sum.cuh), which
// add up in any order: a lane keeps its own smallest exponent (over the three
// channels together) and rescales its sums when a group brings a smaller one,
// and the lanes' sums meet at the run's smallest, emin.  False where the run
// leaves the exact range.  The warp's lanes call it together.
template <int LANES>
__device__ __forceinline__ bool run_sums(const uint32_t* __restrict__ pix, const float* __restrict__ L, uint32_t j0,
                                         uint32_t j1, int c, long long (&acc)[3], int& emin) {
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int STEP = LANES * VU;
    const int count = (int)(j1 - j0);                        // under 2^31 pixels
#pragma unroll
    for (int k = 0; k < 3; ++k) acc[k] = 0;
    emin = fipt_exact::EMPTY_EMIN;
    fipt_exact::Range run;
    bool ok = fipt_exact::spread_limit(count) >= 0;
    uint32_t qn[VU];
#pragma unroll
    for (int u = 0; u < VU; ++u) {
        const uint32_t e = j0 + c + u * LANES;
        qn[u] = e < j1 ? pix[e] : 0u;
    }
    for (uint32_t e = j0 + c; e < j1 && ok; e += STEP) {
        float v[VU][3];
#pragma unroll
        for (int u = 0; u < VU; ++u) {
            const int64_t q = 3 * (int64_t)qn[u];
            const bool in = e + u * LANES < j1;
            v[u][0] = in ? L[q] : 0.0f;
            v[u][1] = in ? L[q + 1] : 0.0f;
            v[u][2] = in ? L[q + 2] : 0.0f;
        }
#pragma unroll
        for (int u = 0; u < VU; ++u) {
            const uint32_t x = e + STEP + u * LANES;
            qn[u] = x < j1 ? pix[x] : 0u;
        }
#pragma unroll
        for (int u = 0; u < VU; ++u)
#pragma unroll
            for (int k = 0; k < 3; ++k) run.note(v[u][k]);
        const int em = run.emin();
        if (em < emin) {            // from EMPTY_EMIN the sums are still 0
            const int sh = min(emin - em, 63);
#pragma unroll
            for (int k = 0; k < 3; ++k) acc[k] = (long long)((unsigned long long)acc[k] << sh);
            emin = em;
        }
        ok = !run.special() && run.exact_for(count);
        if (ok) {
#pragma unroll
            for (int u = 0; u < VU; ++u)
#pragma unroll
                for (int k = 0; k < 3; ++k) acc[k] = fipt_exact::add_term(acc[k], v[u][k], emin);
        }
    }
    if (LANES == 1) return ok;
    // the run's range and sums over its lanes
#pragma unroll
    for (int o = 1; o < LANES; o <<= 1) {
        run.lo = min(run.lo, __shfl_xor_sync(FULL, run.lo, o));
        run.hi = max(run.hi, __shfl_xor_sync(FULL, run.hi, o));
    }
    const unsigned lanes = ((1u << LANES) - 1u) << (threadIdx.x & 31 & ~(LANES - 1));
    ok = (__ballot_sync(FULL, ok) & lanes) == lanes && !run.special() && run.exact_for(count);
    const int sh = ok ? emin - run.emin() : 0;             // 0 to 29 where the lane has a nonzero value
    emin = run.emin();
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        acc[k] = acc[k] == 0 ? 0 : (long long)((unsigned long long)acc[k] << min(sh, 63));
#pragma unroll
        for (int o = 1; o < LANES; o <<= 1) acc[k] += __shfl_xor_sync(FULL, acc[k], o);
    }
    return ok;
}

// Means of the runs.  Long runs take MEAN_LANES lanes each, as the kernel is
// bound by its longest ones (4,194,304 pixels of the room in 256^3 cells, 14 a
// run: 210 us with a lane per run, 17 % of the warps active -> 62 us), then by
// the gathers.  Where MEAN_THREADS neighbouring runs are short most of those
// lanes would idle, and one of their MEAN_SUBS blocks takes them all, a lane each,
// and then the long ones among them as before (4,000,000 points in 256^3 cells,
// 1.1 a run: the whole call 903 us with MEAN_LANES for all, 546 with a lane for
// all, 508).  The choice is made by neighbourhood, as dense cells lie side by side
// and a block that took 128 long runs would work them off one after the other
// (813,120 pixels of a floor in 256^3 cells, 4.2 a run and up to 1,447: 206 us with
// MEAN_LANES for all, 258 with a lane for all under 32 pixels, 201).  MEAN_SHORT 3 /
// 4 / 6 / 8 over 118 calls of 1 to 70 pixels a run: on average 1.03 / 1.05 / 1.05 / 1.05
// times as fast as the faster of one kind for all, at worst 0.98 / 0.99 / 0.97 / 0.95.
//
// Runs outside the exact range are listed by their block, which then adds up
// ten of them a warp, every lane a channel of one, in FP64 in pixel order
// (4,194,304 points in 64^3 cells, all outside it: 403 us with a lane a run, 480
// with three lanes of MEAN_LANES, 400).
__global__ void __launch_bounds__(MEAN_THREADS)
k_vox_means(const uint32_t* __restrict__ keys, const uint32_t* __restrict__ pix, const uint32_t* __restrict__ heads,
            const uint32_t* __restrict__ nhead, const float* __restrict__ L, float4* __restrict__ grid) {
    constexpr unsigned FULL = 0xffffffffu;
    __shared__ uint2 wide[MEAN_THREADS];                   // [j0, j1) of the block's runs outside the exact range
    __shared__ int n_wide;
    const int nh = (int)*nhead, units = (nh + MEAN_UNIT - 1) / MEAN_UNIT;
    const int lane = threadIdx.x & 31, c = lane % MEAN_LANES;
    if (threadIdx.x == 0) n_wide = 0;
    __syncthreads();
    for (int u = blockIdx.x; u < units; u += gridDim.x) {
        // the block's neighbourhood, and which of its blocks works where it is short (another one in each, so that a
        // block that goes round several times works in one of MEAN_SUBS)
        const int near = u / MEAN_SUBS, n0 = near * MEAN_THREADS, n1 = min(nh, n0 + MEAN_THREADS);
        int h = u * MEAN_UNIT + (int)threadIdx.x / MEAN_LANES;
        uint32_t j0 = h < n1 ? heads[h] : 0, j1 = h < n1 ? heads[h + 1] : 0;     // empty past n1
        const bool lanes = heads[n1] - heads[n0] <= (uint32_t)(MEAN_SHORT * (n1 - n0));
        if (lanes) {
            if (u % MEAN_SUBS != near % min(MEAN_SUBS, units - near * MEAN_SUBS)) continue;      // whole block
            h = n0 + (int)threadIdx.x;
            j0 = h < n1 ? heads[h] : 0;
            j1 = h < n1 ? heads[h + 1] : 0;
        }
        const auto group = [&](uint32_t r0, uint32_t r1) {
            long long acc[3];
            int emin;
            const bool ok = run_sums<MEAN_LANES>(pix, L, r0, r1, c, acc, emin);
            if (r1 > r0 && ok && c < 4) {                  // lanes 0 to 2 divide a channel each
                const double s = fipt_exact::scaled_double(c == 0 ? acc[0] : c == 1 ? acc[1] : acc[2], emin);
                reinterpret_cast<float*>(grid + keys[r0])[c] = c < 3 ? (float)(s / (double)(r1 - r0)) : (float)(r1 - r0);
            }
            if (r1 > r0 && !ok && c == 0) wide[atomicAdd(&n_wide, 1)] = make_uint2(r0, r1);
        };
        if (!lanes) {
            group(j0, j1);
        } else {
            const bool is_long = j1 - j0 >= 32;
            long long acc[3];
            int emin;
            const bool ok = run_sums<1>(pix, L, j0, is_long ? j0 : j1, 0, acc, emin);
            if (j1 > j0 && !is_long) {
                if (ok) {
                    const double n = (double)(j1 - j0);
                    grid[keys[j0]] = make_float4((float)(fipt_exact::scaled_double(acc[0], emin) / n),
                                                 (float)(fipt_exact::scaled_double(acc[1], emin) / n),
                                                 (float)(fipt_exact::scaled_double(acc[2], emin) / n), (float)n);
                } else {
                    wide[atomicAdd(&n_wide, 1)] = make_uint2(j0, j1);
                }
            }
            for (unsigned todo = __ballot_sync(FULL, is_long); todo;) {      // four of the long ones
                int of = -1;
#pragma unroll
                for (int g = 0; g < 32 / MEAN_LANES; ++g) {
                    if (lane / MEAN_LANES == g) of = __ffs(todo) - 1;
                    todo &= todo - 1;
                }
                const uint32_t r0 = __shfl_sync(FULL, j0, of & 31), r1 = __shfl_sync(FULL, j1, of & 31);
                group(r0, of < 0 ? r0 : r1);
            }
        }
        __syncthreads();
        const int listed = n_wide, of = lane / 3, ch = lane - 3 * of;
        for (int k = 10 * (threadIdx.x >> 5) + of; k < listed && of < 10; k += 10 * (MEAN_THREADS / 32)) {
            const uint2 run = wide[k];
            double s = 0.0;
            uint32_t e = run.x;
            for (; e + VU <= run.y; e += VU) {
                float v[VU];
#pragma unroll
                for (int q = 0; q < VU; ++q) v[q] = L[3 * (int64_t)pix[e + q] + ch];
#pragma unroll
                for (int q = 0; q < VU; ++q) s += (double)v[q];
            }
            for (; e < run.y; ++e) s += (double)L[3 * (int64_t)pix[e] + ch];
            float* g = reinterpret_cast<float*>(grid + keys[run.x]);
            g[ch] = (float)(s / (double)(run.y - run.x));
            if (ch == 0) g[3] = (float)(run.y - run.x);
        }
        if (u + (int)gridDim.x >= units) break;
        __syncthreads();                                   // the list is read
        if (threadIdx.x == 0) n_wide = 0;
        __syncthreads();
    }
}

struct VoxLayout {
    uint32_t *keys, *keys_alt, *vals, *vals_alt, *hist, *heads, *nhead, *tcount;
    size_t bytes;
};

VoxLayout carve(void* ws, int64_t P) {
    Carver c{static_cast<char*>(ws), 0};
    VoxLayout L;
    const int64_t p1 = P > 0 ? P : 1;
    L.keys = c.take<uint32_t>((size_t)p1);
    L.keys_alt = c.take<uint32_t>((size_t)p1);
    L.vals = c.take<uint32_t>((size_t)p1);
    L.vals_alt = c.take<uint32_t>((size_t)p1);
    L.hist = c.take<uint32_t>(radix_sort_scratch_bytes(p1) / sizeof(uint32_t));
    L.heads = c.take<uint32_t>((size_t)p1 + 1);
    L.nhead = c.take<uint32_t>(1);
    L.tcount = c.take<uint32_t>((size_t)((p1 + HEAD_TILE - 1) / HEAD_TILE));
    L.bytes = c.off + 256;
    return L;
}

inline unsigned blocks(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

extern "C" fipt_status fipt_voxel_cache_workspace_size(int64_t P, size_t* bytes) {
    FIPT_REQUIRE(bytes && P >= 0 && P < ((int64_t)1 << 31), "bad arguments");
    *bytes = carve(nullptr, P).bytes;
    return FIPT_OK;
}

extern "C" fipt_status fipt_voxel_cache_build(fipt_scene* s, const float* x, int64_t x_stride,
                                              const float* L, int64_t P, int32_t R, float* grid,
                                              void* ws, size_t ws_bytes, fipt_stream stream) {
    FIPT_REQUIRE(s, "scene is NULL");
    FIPT_REQUIRE(R >= 1 && R <= 1024, "R must be in [1, 1024]");
    FIPT_REQUIRE(P >= 0 && P < ((int64_t)1 << 31) && x_stride >= 3, "bad sizes");
    FIPT_REQUIRE(grid && fipt_aligned(grid, 16), "grid must be 16-byte aligned");
    FIPT_REQUIRE(P == 0 || (x && L && fipt_aligned(x, 4) && fipt_aligned(L, 4)), "x / L NULL or misaligned");
    VoxLayout Y = carve(ws, P);
    if (!ws || ws_bytes < Y.bytes || !fipt_aligned(ws, 256))
        return fipt_set_error(FIPT_ERR_WORKSPACE, "voxel workspace %zu < %zu bytes (256-aligned)",
                              ws_bytes, Y.bytes);
    FIPT_CUDA(cudaSetDevice(s->ctx->device));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int64_t nv = (int64_t)R * R * R;
    FIPT_CUDA(cudaMemsetAsync(grid, 0, sizeof(float4) * (size_t)nv, st));
    if (P == 0) return FIPT_OK;
    FIPT_LAUNCH(k_vox_keys, blocks(P, 256), 256, 0, st, x, x_stride, P, s->cst, R, Y.keys, Y.vals);
    int bits = 0;
    while (((int64_t)1 << bits) < nv) ++bits;
    bits = (bits + 7) & ~7;
    uint32_t *sk, *sv;
    fipt_status r = radix_sort_pairs<uint32_t>(Y.keys, Y.keys_alt, Y.vals, Y.vals_alt, Y.hist, P,
                                               bits > 0 ? bits : 8, st, &sk, &sv);
    if (r != FIPT_OK) return r;
    const int64_t nt = (P + HEAD_TILE - 1) / HEAD_TILE;
    FIPT_LAUNCH(k_vox_count, (unsigned)nt, HEAD_TILE, 0, st, sk, P, Y.tcount);
    FIPT_LAUNCH(k_vox_scan, 1, HEAD_TILE, 0, st, Y.tcount, nt, Y.heads, Y.nhead, P);
    FIPT_LAUNCH(k_vox_compact, (unsigned)nt, HEAD_TILE, 0, st, sk, P, Y.tcount, Y.heads);
    // a thread per pixel: a unit a block where runs have MEAN_LANES pixels, up to MEAN_SUBS where they have one; an odd
    // multiple of MEAN_SUBS blocks, so that a block's units lie in neighbourhoods of all residues
    const int64_t eighth = (P + MEAN_THREADS * MEAN_SUBS - 1) / (MEAN_THREADS * MEAN_SUBS) | 1;
    FIPT_LAUNCH(k_vox_means, (unsigned)(MEAN_SUBS * eighth), MEAN_THREADS, 0, st, sk, sv, Y.heads, Y.nhead, L,
                reinterpret_cast<float4*>(grid));
    FIPT_LAUNCHED("voxel cache build");
    return FIPT_OK;
}

extern "C" fipt_status fipt_scene_set_voxel_cache(fipt_scene* s, const float* grid, int32_t R) {
    FIPT_REQUIRE(s, "scene is NULL");
    if (!grid) {
        s->vox = nullptr;
        s->vox_r = 0;
        return FIPT_OK;
    }
    FIPT_REQUIRE(R >= 1 && R <= 1024 && fipt_aligned(grid, 16), "bad voxel grid");
    s->vox = reinterpret_cast<const float4*>(grid);
    s->vox_r = R;
    return FIPT_OK;
}
