// Per-triangle rendering error (Sec. 4.4): rendering without the emission
// term leaves large error exactly where the emitters are.  Pixels are
// grouped by their first-hit triangle with a stable radix sort, and the
// squared errors are summed in FP64 over the sorted pixels: a warp takes a
// tile of TILE consecutive ones, row by row, with a segmented scan per row,
// and the segments that cross tiles are joined from the tiles' parts in
// order.  Every sum has a fixed order, so the result is deterministic.
#include "fipt_internal.cuh"

namespace {

__global__ void k_tri_keys(const int32_t* __restrict__ tri, int64_t stride, int64_t P, int64_t T,
                           uint32_t* __restrict__ keys, uint32_t* __restrict__ vals) {
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= P) return;
    const int32_t t = tri[p * stride];
    keys[p] = (t >= 0 && t < T) ? (uint32_t)t : (uint32_t)T;   // T = "no triangle", sorts last
    vals[p] = (uint32_t)p;
}

// A float as a double by integer operations (FP64 conversions run at the rate
// of FP64 additions); subnormals, infinities and NaNs are converted.
__device__ __forceinline__ double widen(float f) {
    const uint32_t b = __float_as_uint(f);
    if (((b >> 23) & 0xffu) - 1u < 254u)
        return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
    return (b << 1) == 0u ? __hiloint2double((int)b, 0) : (double)f;
}

// One warp per TILE sorted pixels.  The kernel is bound by FP64 (1/64 of the
// float32 rate), so its lanes are pixels, all of them busy: 12 FP64
// instructions per row of 32 pixels, however long the segments are.  (A warp
// per triangle spent five additions of its butterfly on each of the floor's
// 2,045,464 triangles, most of them unseen, and a lane of it 3,000 dependent
// gathers on a triangle that 100,000 pixels see: 2,636 us for 4,194,304
// pixels against 153 us here, 107 since the floats widen by integer operations.)
//
// A segment inside the tile is written at its last pixel.  head_sum / head_end
// [w]: the part in tile w of a segment that began before it, and the position
// after its last pixel (-1: it goes on past the tile).  tail_sum / tail_start
// [w]: the part in tile w of a segment that begins in it and goes on, and its
// first position (tail_start -1: none).
constexpr int TILE = 256;

__global__ void __launch_bounds__(256)
k_tile_sums(const uint32_t* __restrict__ keys, const uint32_t* __restrict__ pix, int64_t P, int64_t T,
            const float* __restrict__ Lr, const float* __restrict__ Lgt, double* __restrict__ err,
            int32_t* __restrict__ count, double* __restrict__ head_sum, int32_t* __restrict__ head_end,
            double* __restrict__ tail_sum, int32_t* __restrict__ tail_start) {
    constexpr unsigned FULL = 0xffffffffu;
    constexpr uint32_t NONE = 0xffffffffu;                 // no key: keys are at most T < 2^31 - 1
    const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    const int64_t base = w * TILE;
    if (base >= P) return;                                 // whole warp
    uint32_t prev = base > 0 ? keys[base - 1] : NONE;
    int64_t open = -1;                 // where the segment open at the end of the last row began (-1: before the tile)
    double carry = 0.0;                // its sum in this tile
    bool goes_on = false;
    for (int r = 0; r < TILE / 32; ++r) {
        const int64_t row = base + 32 * r, j = row + lane;
        if (row >= P) break;
        const uint32_t k = j < P ? keys[j] : NONE;
        uint32_t up = __shfl_up_sync(FULL, k, 1), down = __shfl_down_sync(FULL, k, 1);
        if (lane == 0) up = prev;
        if (lane == 31) down = j + 1 < P ? keys[j + 1] : NONE;
        double v = 0.0;
        if (k < (uint32_t)T) {
            const int64_t p = pix[j];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const double d = widen(Lr[3 * p + c]) - widen(Lgt[3 * p + c]);
                v = fma(d, d, v);
            }
        }
        const unsigned heads = __ballot_sync(FULL, k != up);
        const unsigned mine = heads & (FULL >> (31 - lane));
        const int first = mine ? 31 - __clz(mine) : 0;     // the row's first lane of this lane's segment
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double y = __shfl_up_sync(FULL, v, o);
            if (lane - o >= first) v += y;
        }
        if (mine == 0) v += carry;
        if (k < (uint32_t)T && k != down) {                // the segment's last pixel
            const int64_t start = mine ? row + first : open;
            if (start >= 0) {
                err[k] = v;
                count[k] = (int32_t)(j + 1 - start);
            } else {
                head_sum[w] = v;
                head_end[w] = (int32_t)(j + 1);
            }
        }
        prev = __shfl_sync(FULL, k, 31);
        carry = __shfl_sync(FULL, v, 31);
        goes_on = __shfl_sync(FULL, k < (uint32_t)T && k == down ? 1 : 0, 31) != 0;
        if (heads) open = row + 31 - __clz(heads);
    }
    if (lane == 0) {
        tail_start[w] = goes_on ? (int32_t)open : -1;
        if (goes_on && open >= 0) tail_sum[w] = carry;
        if (goes_on && open < 0) {
            head_sum[w] = carry;
            head_end[w] = -1;
        }
    }
}

// The segments that cross tiles: a thread per tile in which one begins, its
// warp for one that spans whole tiles.
__global__ void __launch_bounds__(256)
k_join_tiles(const uint32_t* __restrict__ keys, int64_t tiles, const double* __restrict__ head_sum,
             const int32_t* __restrict__ head_end, const double* __restrict__ tail_sum,
             const int32_t* __restrict__ tail_start, double* __restrict__ err, int32_t* __restrict__ count) {
    constexpr unsigned FULL = 0xffffffffu;
    const int64_t w = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    const int32_t start = w + 1 < tiles ? tail_start[w] : -1;
    int32_t end = start >= 0 ? head_end[w + 1] : 0;
    double rest = start >= 0 && end >= 0 ? head_sum[w + 1] : 0.0;
    for (unsigned todo = __ballot_sync(FULL, end < 0); todo; todo &= todo - 1) {
        const int l = __ffs(todo) - 1;
        double s = 0.0;
        for (int64_t i = __shfl_sync(FULL, w, l) + 1 + lane;; i += 32) {
            const int32_t e = i < tiles ? head_end[i] : 0;
            const unsigned m = __ballot_sync(FULL, e >= 0);
            const int last = m ? __ffs(m) - 1 : 31;
            if (lane <= last && i < tiles) s += head_sum[i];
            if (m) {
                const int32_t at = __shfl_sync(FULL, e, last);
                if (lane == l) end = at;
                break;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
        if (lane == l) rest = s;
    }
    if (start >= 0) {
        const uint32_t k = keys[(w + 1) * TILE - 1];
        err[k] = tail_sum[w] + rest;
        count[k] = end - start;
    }
}

struct TriErrLayout {
    uint32_t *keys, *keys_alt, *vals, *vals_alt, *hist;
    double *head_sum, *tail_sum;
    int32_t *head_end, *tail_start;
    int64_t tiles;
    size_t bytes;
};

TriErrLayout carve(void* ws, int64_t P) {
    Carver c{static_cast<char*>(ws), 0};
    TriErrLayout L;
    const int64_t p1 = P > 0 ? P : 1;
    L.keys = c.take<uint32_t>((size_t)p1);
    L.keys_alt = c.take<uint32_t>((size_t)p1);
    L.vals = c.take<uint32_t>((size_t)p1);
    L.vals_alt = c.take<uint32_t>((size_t)p1);
    L.hist = c.take<uint32_t>(radix_sort_scratch_bytes(p1) / sizeof(uint32_t));
    L.tiles = (p1 + TILE - 1) / TILE;
    L.head_sum = c.take<double>((size_t)L.tiles);
    L.tail_sum = c.take<double>((size_t)L.tiles);
    L.head_end = c.take<int32_t>((size_t)L.tiles);
    L.tail_start = c.take<int32_t>((size_t)L.tiles);
    L.bytes = c.off + 256;
    return L;
}

inline unsigned blocks(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

extern "C" fipt_status fipt_tri_error_workspace_size(int64_t P, int64_t T, size_t* bytes) {
    FIPT_REQUIRE(bytes && P >= 0 && T >= 0 && P < ((int64_t)1 << 31) && T < ((int64_t)1 << 31) - 1,
                 "bad arguments");
    *bytes = carve(nullptr, P).bytes;
    return FIPT_OK;
}

extern "C" fipt_status fipt_tri_error(const int32_t* tri, int64_t tri_stride, const float* Lr,
                                      const float* Lgt, int64_t P, int64_t T, double* err_sum, int32_t* count, void* ws,
                                      size_t ws_bytes, fipt_stream stream) {
    FIPT_REQUIRE(P >= 0 && T >= 0 && P < ((int64_t)1 << 31) && T < ((int64_t)1 << 31) - 1,
                 "bad sizes P=%lld T=%lld", (long long)P, (long long)T);
    FIPT_REQUIRE(tri_stride >= 1, "tri_stride must be >= 1");
    if (T == 0) return FIPT_OK;
    FIPT_REQUIRE(err_sum && count && fipt_aligned(err_sum, 8) && fipt_aligned(count, 4),
                 "err_sum / count NULL or misaligned");
    FIPT_REQUIRE(P == 0 || (tri && Lr && Lgt && fipt_aligned(tri, 4) && fipt_aligned(Lr, 4) &&
                            fipt_aligned(Lgt, 4)), "tri / Lr / Lgt NULL or misaligned");
    TriErrLayout L = carve(ws, P);
    if (!ws || ws_bytes < L.bytes || !fipt_aligned(ws, 256))
        return fipt_set_error(FIPT_ERR_WORKSPACE, "tri_error workspace %zu < %zu bytes (256-aligned)",
                              ws_bytes, L.bytes);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    FIPT_CUDA(cudaMemsetAsync(err_sum, 0, sizeof(double) * (size_t)T, st));      // triangles no pixel sees
    FIPT_CUDA(cudaMemsetAsync(count, 0, sizeof(int32_t) * (size_t)T, st));
    if (P > 0) {
        uint32_t* sk = L.keys;
        uint32_t* sv = L.vals;
        FIPT_LAUNCH(k_tri_keys, blocks(P, 256), 256, 0, st, tri, tri_stride, P, T, L.keys, L.vals);
        int bits = 0;
        while (((int64_t)1 << bits) <= T) ++bits;      // keys lie in [0, T]
        bits = (bits + 7) & ~7;
        fipt_status r = radix_sort_pairs<uint32_t>(L.keys, L.keys_alt, L.vals, L.vals_alt, L.hist, P,
                                                   bits, st, &sk, &sv);
        if (r != FIPT_OK) return r;
        FIPT_LAUNCH(k_tile_sums, blocks(L.tiles * 32, 256), 256, 0, st, sk, sv, P, T, Lr, Lgt, err_sum, count,
                    L.head_sum, L.head_end, L.tail_sum, L.tail_start);
        FIPT_LAUNCH(k_join_tiles, blocks(L.tiles, 256), 256, 0, st, sk, L.tiles, L.head_sum, L.head_end, L.tail_sum,
                    L.tail_start, err_sum, count);
    }
    FIPT_LAUNCHED("tri_error");
    return FIPT_OK;
}
