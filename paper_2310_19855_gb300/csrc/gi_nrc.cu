// Learned radiance surrogate: multiresolution hash encoding (Mueller et al. 2022) of the hit
// position and normal direction code, a 32 -> 64 -> 64 -> 3 ReLU network without bias terms on the
// fifth-generation tensor cores (tcgen05 MMAs from shared memory into tensor memory), relative-L2
// loss (Mueller et al. 2021) and Adam (Kingma and Ba 2015), trained online on the world cache's
// resolved cells.  The paper itself has no learned part.
//
// Passes of one training step (all on the caller's stream):
//   k_nrc_encode   one thread per (sample, level): normalise the position, find the level's cell,
//                  gather the 8 vertices' float16 features, interpolate, write the sample's row of
//                  the bf16 input tile (and its target / mask plane, and record index)
//   k_nrc_mlp      persistent, one CTA per SM, 128-sample tiles: forward, loss gradient, backward
//                  through the three layers, weight gradients accumulated in tensor memory over all
//                  the CTA's tiles, input gradients out to global memory
//   k_nrc_scatter  one thread per (sample, level): trilinear weights x input gradient added to the
//                  8 vertices' gradient accumulators (float2 atomics)
//   k_nrc_adam     Adam on the table entries and the weights (with the network kernel's partial weight
//                  gradients summed); refreshes the float16 table copy and the bf16 weight images
//                  the MLP kernel loads
//
// Shared-memory operand layout: see gi_tc.cuh (K-major core matrices, no swizzle).  Every tile of
// the MLP kernel is stored sample-major; the weight-gradient products, which contract over the
// samples, read the same tiles through MN-major descriptors (LBO = stride between 8-sample groups,
// SBO = stride between 8-feature groups), so no tile is ever transposed.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <vector>

#include "gi_internal.cuh"
#include "gi_tc.cuh"

namespace gi {
namespace {

constexpr int kL = GI_NRC_LEVELS;    // 16 levels
constexpr int kIn = 2 * kL;          // 32 encoded features
constexpr int kHid = GI_NRC_HIDDEN;  // 64 hidden units
constexpr int kOut = GI_NRC_OUTPUTS; // 3 outputs
constexpr int kTile = 128;           // samples per tile = M of every forward / backward product
constexpr int kEncThreads = 256, kEncBlocksPerSm = 5;
constexpr uint32_t kPrimeY = 2654435761u, kPrimeZ = 805459861u, kPrimeD = 2246822519u;

// bf16 weight images (core-matrix tiles), loaded into shared memory by every MLP CTA
constexpr uint32_t kImgW1 = 0;        // W1   [64 out][32 in]   SBO 512
constexpr uint32_t kImgW1T = 4096;    // W1^T [32 in][64 out]   SBO 1024
constexpr uint32_t kImgW2 = 8192;     // W2   [64][64]          SBO 1024
constexpr uint32_t kImgW2T = 16384;   // W2^T [64][64]          SBO 1024
constexpr uint32_t kImgW3P = 24576;   // W3   [16 out][64 in]   SBO 1024, rows 3..15 zero
constexpr uint32_t kImgW3PT = 26624;  // W3^T [64 in][16 out]   SBO 256, columns 3..15 zero
constexpr uint32_t kImgBytes = 28672;

// float32 master weights: W1 | W2 | W3, row-major [out][in]
constexpr int kW1 = 0, kW2 = kHid * kIn, kW3 = kW2 + kHid * kHid, kWCount = kW3 + kOut * kHid;
// a CTA's partial: the weight gradients of its tiles, then its loss, sum m|y - t|, sum m|t|
constexpr int kPartStride = kWCount + 4;

// global input tile: [128 samples][32 features] bf16 core matrices; 8-sample group g = bytes 512 g ..
constexpr uint32_t kXTile = kTile * kIn * 2;  // 8192
constexpr uint32_t kTTile = 4 * kTile * 4;    // target planes r, g, b and the mask: 2048

// training kernel shared memory (bytes)
constexpr uint32_t kSmImg = 0;
constexpr uint32_t kSmXH0 = 28672;   // [128][96]: H1 (features 0..63) | X (64..95), SBO 1536
constexpr uint32_t kSmXH1 = 53248;
constexpr uint32_t kSmT0 = 77824;    // target tiles
constexpr uint32_t kSmT1 = 79872;
constexpr uint32_t kSmH2 = 81920;    // [128][64], SBO 1024
constexpr uint32_t kSmDY = 98304;    // [128][16], SBO 256
constexpr uint32_t kSmZ = 102400;    // [128][128]: dZ2 (0..63) | dZ1 (64..127), SBO 2048
constexpr uint32_t kSmTrain = 135168;
constexpr uint32_t kXHStride = 1536, kH2Stride = 1024, kDYStride = 256, kZStride = 2048;

// tensor memory columns (256 allocated)
constexpr uint32_t kTmD1 = 0;    // layer-1 pre-activation, then dH1, then dX
constexpr uint32_t kTmD2 = 64;   // layer-2 pre-activation, then dH2
constexpr uint32_t kTmD3 = 128;  // output (16 columns, 3 used)
constexpr uint32_t kTmGC = 144;  // dW3^T accumulator (16 columns)
constexpr uint32_t kTmGA = 160;  // [dW2 | dW1] accumulator (96 columns)
constexpr uint32_t kTmCols = 256;

// inference kernel: shared memory (W1, W2 and W3 of the image, two input tiles, one tile of hidden
// units) and tensor memory small enough for four CTAs per SM
constexpr uint32_t kInfW1 = 0, kInfW2 = 4096, kInfW3 = 12288, kInfX = 14336, kInfH = 30720, kInfBytes = 47104;
constexpr uint32_t kInfCols = 128, kInfD = 0, kInfD3 = 64;

constexpr uint32_t kErrTimeout = 1u;

// One table entry: float32 master features and Adam moments, padded to one sector.  The
// gradient accumulators live in a separate dense float2 array, so that the Adam pass can find
// the entries a step touched with one coalesced 8-byte read per entry.
struct __align__(32) Entry {
    float2 p, m, v, pad;
};
static_assert(sizeof(Entry) == 32, "entry must fill one sector");

struct Levels {
    uint32_t res[kL];
    uint32_t dense[kL];
};

struct Geometry {
    float lo[3], inv_ext[3];
    Levels lv;
    uint32_t log2_table;
};

enum EncMode { kEncPoints = 0, kEncSampled = 1 };  // of k_nrc_encode

struct EncArgs {
    Geometry geo;
    const __half2 *tab16;
    // points (kEncPoints) or records (kEncSampled, k_nrc_encode_queries)
    const float *pos[3];
    const float *nrm[3];
    const float *len;          // records: ray length (hit test)
    uint32_t n;                // samples (points / batch); queries: capacity
    const float *target[3];    // kEncPoints training targets (or NULL)
    const float *mask;         // kEncPoints sample mask (or NULL = 1)
    // kEncSampled: sample s of the launch is sample offset + s of the frame
    uint32_t n_records, seed, offset;
    const uint32_t *slot_ids;
    CacheView cv;
    // k_nrc_encode_queries
    const uint32_t *qidx;
    const uint32_t *qcount;
    // outputs
    uint16_t *X;               // input tiles
    float *T;                  // target tiles (NULL when not training)
    uint32_t *idx;             // record index per sample (kEncSampled)
};

struct MlpArgs {
    const uint16_t *X;
    const float *T;
    const uint8_t *wimg;
    uint32_t n;                // samples
    float dy_scale;            // 2 / B
    float loss_eps;
    float *dX;                 // [n_pad][32] float32
    float *wpart;              // per-CTA partial W1 | W2 | W3 gradients and loss sums, rows of
                               // kPartStride floats (summed by k_nrc_adam or k_nrc_wgrad_reduce)
    uint32_t *err;
};

struct InferArgs {
    const uint16_t *X;
    const uint8_t *wimg;
    uint32_t n;                // samples, unless count is given
    const uint32_t *count;     // device sample count (queries), clamped to n
    float4 *out;               // (max(y, 0), 1)
    const uint32_t *out_idx;   // out[out_idx[s]] when given, else out[s]
    uint32_t *err;
};

struct ScatterArgs {
    Geometry geo;
    const float *pos[3];
    const float *nrm[3];
    const uint32_t *idx;       // record of each sample (NULL: sample s is point s)
    uint32_t n;
    const float *dX;
    float2 *grad;
};

struct SelectArgs {
    const float *pos[3];
    const float *len;
    const uint32_t *slot_ids;
    uint32_t n;
    CacheView cv;
    KeyParams kp;
    uint32_t query_lod;
    float trust;
    uint32_t trained;
    const float *stats;
    uint32_t max_q;
    uint32_t *qidx;
    uint32_t *qcount;
    uint32_t *bits;
};

// ---------------------------------------------------------------- encoding

// dominant axis of the normal (ties x, then y) and the sign bit of that component
__device__ __forceinline__ uint32_t dir_code(float nx, float ny, float nz) {
    const float ax = fabsf(nx), ay = fabsf(ny), az = fabsf(nz);
    const int axis = (ax >= ay && ax >= az) ? 0 : (ay >= az ? 1 : 2);
    const float comp = axis == 0 ? nx : (axis == 1 ? ny : nz);
    return 2u * (uint32_t)axis + (__float_as_uint(comp) >> 31);
}

// Table indices (within the level) and trilinear weights of the 8 vertices around a point.
// Corner c has offsets (c & 1, c >> 1 & 1, c >> 2 & 1).  x: normalised position in [0, 1]^3.
__device__ __forceinline__ void level_corners(const float (&x)[3], uint32_t R, bool dense, uint32_t d,
                                              uint32_t tmask, uint32_t (&idx)[8], float (&w)[8]) {
    uint32_t i[3];
    float f[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float s = __fmul_rn(x[a], (float)R);
        const int ii = min(__float2int_rd(s), (int)R - 1);
        i[a] = (uint32_t)ii;
        f[a] = __fsub_rn(s, (float)ii);
    }
    const uint32_t V = R + 1u;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const uint32_t vx = i[0] + (c & 1), vy = i[1] + ((c >> 1) & 1), vz = i[2] + ((c >> 2) & 1);
        idx[c] = dense ? ((d * V + vz) * V + vy) * V + vx : ((vx ^ (vy * kPrimeY) ^ (vz * kPrimeZ) ^ (d * kPrimeD)) & tmask);
        const float wx = (c & 1) ? f[0] : 1.0f - f[0];
        const float wy = ((c >> 1) & 1) ? f[1] : 1.0f - f[1];
        const float wz = ((c >> 2) & 1) ? f[2] : 1.0f - f[2];
        w[c] = wx * wy * wz;
    }
}

__device__ __forceinline__ void normalise(const Geometry &g, float px, float py, float pz, float (&x)[3]) {
    const float p[3] = {px, py, pz};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        // fmaxf turns NaN into 0
        x[a] = fminf(fmaxf(__fmul_rn(__fsub_rn(p[a], g.lo[a]), g.inv_ext[a]), 0.0f), 1.0f);
    }
}

__device__ __forceinline__ bool record_hit(const float *const pos[3], const float *len, uint32_t r) {
    const float l = __ldca(len + r);
    return isfinite(l) && l >= 0.0f && isfinite(__ldca(pos[0] + r)) && isfinite(__ldca(pos[1] + r)) &&
           isfinite(__ldca(pos[2] + r));
}

__device__ __forceinline__ float4 cache_value(const CacheView &cv, uint32_t s) {
    const char *r = static_cast<const char *>(cv.resolved) + (size_t)s * cv.resolved_stride;
    if (cv.resolved_f16) {
        const ushort4 h = __ldca(reinterpret_cast<const ushort4 *>(r));
        return make_float4(__half2float(__ushort_as_half(h.x)), __half2float(__ushort_as_half(h.y)),
                           __half2float(__ushort_as_half(h.z)), __half2float(__ushort_as_half(h.w)));
    }
    return __ldca(reinterpret_cast<const float4 *>(r));
}

// a cell resolved without history (see store_resolved)
__device__ __forceinline__ bool cache_cold(const CacheView &cv, uint32_t s) {
    if (cv.cold) return (__ldca(cv.cold + (s >> 5)) >> (s & 31u)) & 1u;
    return cache_value(cv, s).w != 0.0f;
}

__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&h);
}


// The features of the 8 vertices, gathered together, then weighted in corner order.
__device__ __forceinline__ void interpolate_level(const __half2 *tab, const uint32_t (&idx)[8], const float (&w)[8],
                                                  float &e0, float &e1) {
    __half2 f[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) f[c] = __ldca(tab + idx[c]);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const float2 v = __half22float2(f[c]);
        e0 = fmaf(w[c], v.x, e0);
        e1 = fmaf(w[c], v.y, e1);
    }
}

// Points and training samples (drawn at random over the view): one thread per sample and level, a warp
// takes two samples.  MODE: kEncPoints or kEncSampled.
template <int MODE>
__global__ void __launch_bounds__(kEncThreads) k_nrc_encode(EncArgs a) {
    const uint32_t bid = blockIdx.x + pass_begin();
    const uint32_t n = a.n;
    const uint32_t n_pad = (n + kTile - 1) / kTile * kTile;
    const uint32_t T = 1u << a.geo.log2_table;
    for (uint32_t i = bid * blockDim.x + threadIdx.x; i < n_pad * kL; i += gridDim.x * blockDim.x) {
        const uint32_t s = i >> 4, l = i & 15u;
        const bool valid = s < n;
        uint32_t r = s;
        if (MODE == kEncSampled) r = pcg_hash((a.offset + s) ^ a.seed) % a.n_records;
        float e0 = 0.0f, e1 = 0.0f;
        if (valid) {
            float x[3];
            normalise(a.geo, __ldca(a.pos[0] + r), __ldca(a.pos[1] + r), __ldca(a.pos[2] + r), x);
            const uint32_t d = dir_code(__ldca(a.nrm[0] + r), __ldca(a.nrm[1] + r), __ldca(a.nrm[2] + r));
            uint32_t idx[8];
            float w[8];
            level_corners(x, a.geo.lv.res[l], a.geo.lv.dense[l] != 0u, d, T - 1u, idx, w);
            interpolate_level(a.tab16 + (size_t)l * T, idx, w, e0, e1);
        }
        const uint32_t tile = s / kTile, row = s % kTile;
        uint8_t *xt = reinterpret_cast<uint8_t *>(a.X) + (size_t)tile * kXTile;
        *reinterpret_cast<__nv_bfloat162 *>(xt + tc::cm_offset(row, 2u * l, kIn)) = __floats2bfloat162_rn(e0, e1);
        if (a.T && l == 0) {
            float t[3] = {0.f, 0.f, 0.f}, m = 0.0f;
            if (valid && MODE == kEncPoints) {
                for (int c = 0; c < 3; ++c) t[c] = __ldca(a.target[c] + s);
                m = a.mask ? __ldca(a.mask + s) : 1.0f;
            }
            if (valid && MODE == kEncSampled) {
                const uint32_t slot = __ldca(a.slot_ids + r);
                if (slot < a.cv.slots && record_hit(a.pos, a.len, r)) {
                    const float4 v = cache_value(a.cv, slot);
                    t[0] = v.x;
                    t[1] = v.y;
                    t[2] = v.z;
                    m = 1.0f;
                }
                a.idx[s] = r;
            }
            float *tt = a.T + (size_t)tile * (kTTile / 4);
            for (int c = 0; c < 3; ++c) tt[c * kTile + row] = t[c];
            tt[3 * kTile + row] = m;
        }
    }
}

// The records a view leaves to the network.  A warp takes 32 consecutive ones through a
// group of consecutive levels, one level at a time: its lanes' vertices then lie in one level's table,
// close together where the records are (they come probe by probe), and each record's position and normal
// are read once per group.  A block takes a contiguous run of such items, so that the records of an
// SM are neighbours too.  The gathers are bound by the sectors the L2 delivers (45 % of them hit the
// L1 with a thread per record and level), so what counts is how many the L1 answers.  Groups of 16, 8, 4
// or 2 levels, the longest whose busiest warp takes at most 8/7 of the fewest levels that any length gives it
// (230,400 records are 1.2 items of 16 levels a warp: the query frame 102 us so, 78 us with 4.7 items of 4);
// fewer records take k_nrc_encode's form.  On the far hits of a 1080p frame the frame took 366, 363 and 396 us on three scenes, against
// 381, 368 and 417 us with k_nrc_encode's form (random samples and points: 3 us slower, so they keep
// theirs).  48 registers, 5 blocks per SM: at 6 blocks the eight gathers of a level no longer fly
// together, 32 us slower.
__global__ void __launch_bounds__(kEncThreads, kEncBlocksPerSm) k_nrc_encode_queries(EncArgs a) {
    const uint32_t bid = blockIdx.x + pass_begin();
    const uint32_t n = min(ld(a.qcount), a.n);
    const uint32_t T = 1u << a.geo.log2_table;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    // log2 of the levels per group
    const uint32_t n_pad = (n + kTile - 1) / kTile * kTile;
    uint32_t glog = 0;
    if (n / 32u * 8u >= gridDim.x * (kEncThreads / 32)) {
        uint32_t best = 0xFFFFFFFFu;
#pragma unroll
        for (uint32_t g = 1; g <= 4; ++g) {
            // levels that the busiest warp takes
            const uint32_t runs = (n_pad / 32u * (kL >> g) + kEncThreads / 32 - 1) / (kEncThreads / 32);
            const uint32_t levels = ((runs + gridDim.x - 1) / gridDim.x) << g;
            if (g == 1 || 7u * levels <= 8u * best) glog = g;
            best = min(best, levels);
        }
    }
    const uint32_t lgs = kL >> glog;  // level groups
    const uint32_t items = glog ? n_pad / 32u * lgs : n_pad / 2u;
    // contiguous runs of 8 items (one per warp) per block, as even as they divide
    const uint32_t rounds = (items + kEncThreads / 32 - 1) / (kEncThreads / 32);
    const uint32_t r0 = (uint32_t)((uint64_t)rounds * bid / gridDim.x),
                   r1 = (uint32_t)((uint64_t)rounds * (bid + 1) / gridDim.x);
    for (uint32_t it = r0 * (kEncThreads / 32) + warp; it < min(items, r1 * (kEncThreads / 32)); it += kEncThreads / 32) {
        const uint32_t s = glog ? (it / lgs) * 32u + lane : it * 2u + (lane >> 4);
        const uint32_t l0 = glog ? (it % lgs) << glog : (lane & 15u);
        const bool valid = s < n;
        float x[3] = {0.f, 0.f, 0.f};
        uint32_t d = 0;
        if (valid) {
            const uint32_t r = __ldca(a.qidx + s);
            normalise(a.geo, __ldca(a.pos[0] + r), __ldca(a.pos[1] + r), __ldca(a.pos[2] + r), x);
            d = dir_code(__ldca(a.nrm[0] + r), __ldca(a.nrm[1] + r), __ldca(a.nrm[2] + r));
        }
        const uint32_t tile = s / kTile, row = s % kTile;
        uint8_t *xt = reinterpret_cast<uint8_t *>(a.X) + (size_t)tile * kXTile;
        uint4 q = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll 1
        for (uint32_t l = l0; l < l0 + (1u << glog); ++l) {
            float e0 = 0.0f, e1 = 0.0f;
            if (valid) {
                uint32_t idx[8];
                float w[8];
                level_corners(x, a.geo.lv.res[l], a.geo.lv.dense[l] != 0u, d, T - 1u, idx, w);
                interpolate_level(a.tab16 + (size_t)l * T, idx, w, e0, e1);
            }
            const uint32_t pk = pack_bf16x2(e0, e1);
            if (glog == 0u) {
                *reinterpret_cast<uint32_t *>(xt + tc::cm_offset(row, 2u * l, kIn)) = pk;
            } else if (glog == 1u) {
                if (l & 1u) *reinterpret_cast<uint2 *>(xt + tc::cm_offset(row, 2u * (l - 1u), kIn)) = make_uint2(q.x, pk);
                else q.x = pk;
            } else {  // four levels fill 16 bytes of the sample's row
                const uint32_t j = l & 3u;
                if (j == 0u) q.x = pk;
                else if (j == 1u) q.y = pk;
                else if (j == 2u) q.z = pk;
                else {
                    q.w = pk;
                    *reinterpret_cast<uint4 *>(xt + tc::cm_offset(row, 2u * (l & ~3u), kIn)) = q;
                }
            }
        }
    }
}

// ---------------------------------------------------------------- the network on the tensor cores

// Store 8 consecutive features (k0 .. k0 + 7) of sample row t as one 16-byte core-matrix row.
__device__ __forceinline__ void store_row8(uint8_t *tile, uint32_t row_stride, uint32_t t, uint32_t k0, const float *v) {
    const uint4 q = make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]), pack_bf16x2(v[4], v[5]),
                               pack_bf16x2(v[6], v[7]));
    *reinterpret_cast<uint4 *>(tile + (t >> 3) * row_stride + (k0 >> 3) * 128u + (t & 7u) * 16u) = q;
}

// 64 accumulator columns of this thread's row
__device__ __forceinline__ void tmem_ld64(uint32_t tmem, uint32_t warp, uint32_t col, float (&z)[64]) {
    float v0[16], v1[16], v2[16], v3[16];
    tc::tmem_ld16(tc::tmem_lane_addr(tmem, warp, col), v0);
    tc::tmem_ld16(tc::tmem_lane_addr(tmem, warp, col + 16), v1);
    tc::tmem_ld16(tc::tmem_lane_addr(tmem, warp, col + 32), v2);
    tc::tmem_ld16(tc::tmem_lane_addr(tmem, warp, col + 48), v3);
    tc::wait_ld();
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        z[j] = v0[j];
        z[16 + j] = v1[j];
        z[32 + j] = v2[j];
        z[48 + j] = v3[j];
    }
}

__device__ __forceinline__ uint32_t idesc_mn(uint32_t M, uint32_t N) {
    return tc::idesc_bf16(M, N) | (1u << 15) | (1u << 16);
}

// Persistent kernel: CTA b takes tiles b, b + gridDim.x, ...; thread t owns sample row t of a tile
// (tensor-memory lane t: warp w reads lanes 32 w .. 32 w + 31).  Thread 0 issues every MMA and
// bulk copy; completion comes back through mbarriers, every wait bounded in time.
__global__ void __launch_bounds__(kTile, 1) k_nrc_mlp(MlpArgs a) {
    const uint32_t bid = blockIdx.x + pass_begin();
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ __align__(8) uint64_t bar_w, bar_ld[2], bar_mma;
    __shared__ uint32_t tmem_s;
    __shared__ int abort_s;
    const uint32_t t = threadIdx.x, warp = t >> 5;
    const uint32_t tiles = (a.n + kTile - 1) / kTile;
    if (bid >= tiles) return;

    if (t == 0) {
        abort_s = 0;
        tc::mbar_init(&bar_w, 1);
        tc::mbar_init(&bar_ld[0], 1);
        tc::mbar_init(&bar_ld[1], 1);
        tc::mbar_init(&bar_mma, 1);
        tc::mbar_init_fence();
    }
    // dY columns 3..15 stay zero; written once here, never again
    for (uint32_t i = t; i < kTile * 16 / 8; i += kTile)
        reinterpret_cast<uint4 *>(smem + kSmDY)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (warp == 0) {
        tc::tmem_alloc(&tmem_s, kTmCols);
        tc::tmem_relinquish();
    }
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = tmem_s;
    const uint32_t sm = tc::smem_u32(smem);
    auto xh_off = [](int buf) { return buf ? kSmXH1 : kSmXH0; };
    auto t_off = [](int buf) { return buf ? kSmT1 : kSmT0; };
    // Thread 0 counts the asynchronous operations it started and the completions it saw, so that
    // a CTA that gives up after a wait ran out first waits (bounded again) for what it still has in
    // flight -- at most one load per buffer and one MMA group -- before freeing its tensor memory.
    uint32_t ld_issued[2] = {0u, 0u}, ld_done[2] = {0u, 0u}, mma_issued = 0u, mma_done = 0u;
    bool w_done = false;

    auto load_tile = [&](uint32_t tile, int buf) {  // thread 0 only
        ++ld_issued[buf];
        tc::mbar_expect_tx(&bar_ld[buf], kXTile + kTTile);
        const uint8_t *src = reinterpret_cast<const uint8_t *>(a.X) + (size_t)tile * kXTile;
        for (uint32_t g = 0; g < kTile / 8; ++g)
            tc::bulk_g2s(smem + xh_off(buf) + g * kXHStride + 1024u, src + g * 512u, 512u, &bar_ld[buf]);
        tc::bulk_g2s(smem + t_off(buf), reinterpret_cast<const uint8_t *>(a.T) + (size_t)tile * kTTile, kTTile,
                     &bar_ld[buf]);
    };
    if (t == 0) {
        tc::mbar_expect_tx(&bar_w, kImgBytes);
        tc::bulk_g2s(smem + kSmImg, a.wimg, kImgBytes, &bar_w);
        load_tile(bid, 0);
    }
    bool ok = tc::mbar_wait(&bar_w, 0);
    w_done = ok;
    uint32_t ph = 0;  // parity of the next MMA completion
    float loss = 0.f, jerr = 0.f, jtgt = 0.f;
    uint32_t it = 0;
    auto commit_mma = [&]() {  // thread 0 only
        tc::commit(&bar_mma);
        ++mma_issued;
    };
    auto mma_wait = [&]() {
        const bool got = tc::mbar_wait(&bar_mma, ph);
        if (got) ++mma_done;
        ok = got && ok;
        ph ^= 1u;
        tc::fence_after_sync();
    };
    auto sync_operands = [&]() {  // generic smem writes -> tensor cores; TMEM reads done
        tc::fence_async_smem();
        tc::fence_before_sync();
        if (!ok) abort_s = 1;
        __syncthreads();
    };

    for (uint32_t tile = bid; tile < tiles; tile += gridDim.x, ++it) {
        const int buf = it & 1;
        const bool got = tc::mbar_wait(&bar_ld[buf], (it >> 1) & 1u);
        if (got) ++ld_done[buf];
        ok = got && ok;
        if (!ok) abort_s = 1;
        __syncthreads();
        if (abort_s) break;
        if (t == 0 && tile + gridDim.x < tiles) load_tile(tile + gridDim.x, buf ^ 1);
        const uint32_t xh = sm + xh_off(buf);
        uint8_t *xh_p = smem + xh_off(buf);

        // ---- layer 1: D1 = X W1^T
        if (t == 0) {
            tc::fence_after_sync();
            for (uint32_t ks = 0; ks < kIn / 16; ++ks)
                tc::mma_bf16(tmem + kTmD1, tc::smem_desc(xh + 1024u + ks * 256u, 128u, kXHStride),
                             tc::smem_desc(sm + kSmImg + kImgW1 + ks * 256u, 128u, 512u), tc::idesc_bf16(128, 64), ks);
            commit_mma();
        }
        mma_wait();
        float z[64];
        uint32_t m1[2] = {0u, 0u}, m2[2] = {0u, 0u};
        tmem_ld64(tmem, warp, kTmD1, z);
#pragma unroll
        for (int j = 0; j < 64; ++j) {
            m1[j >> 5] |= (z[j] > 0.0f ? 1u : 0u) << (j & 31);
            z[j] = fmaxf(z[j], 0.0f);
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) store_row8(xh_p, kXHStride, t, 8u * j, z + 8 * j);
        sync_operands();
        if (abort_s) break;

        // ---- layer 2: D2 = H1 W2^T
        if (t == 0) {
            tc::fence_after_sync();
            for (uint32_t ks = 0; ks < kHid / 16; ++ks)
                tc::mma_bf16(tmem + kTmD2, tc::smem_desc(xh + ks * 256u, 128u, kXHStride),
                             tc::smem_desc(sm + kSmImg + kImgW2 + ks * 256u, 128u, 1024u), tc::idesc_bf16(128, 64), ks);
            commit_mma();
        }
        mma_wait();
        tmem_ld64(tmem, warp, kTmD2, z);
#pragma unroll
        for (int j = 0; j < 64; ++j) {
            m2[j >> 5] |= (z[j] > 0.0f ? 1u : 0u) << (j & 31);
            z[j] = fmaxf(z[j], 0.0f);
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) store_row8(smem + kSmH2, kH2Stride, t, 8u * j, z + 8 * j);
        sync_operands();
        if (abort_s) break;

        // ---- layer 3: D3 = H2 W3^T (16 columns, 3 used)
        if (t == 0) {
            tc::fence_after_sync();
            for (uint32_t ks = 0; ks < kHid / 16; ++ks)
                tc::mma_bf16(tmem + kTmD3, tc::smem_desc(sm + kSmH2 + ks * 256u, 128u, kH2Stride),
                             tc::smem_desc(sm + kSmImg + kImgW3P + ks * 256u, 128u, 1024u), tc::idesc_bf16(128, 16), ks);
            commit_mma();
        }
        mma_wait();
        float y[16];
        tc::tmem_ld16(tc::tmem_lane_addr(tmem, warp, kTmD3), y);
        tc::wait_ld();
        const uint32_t s = tile * kTile + t;

        // ---- loss gradient: dy = m (2 / B) (y - t) / (y^2 + eps); relative L2 and the judge's sums
        const float *tt = reinterpret_cast<const float *>(smem + t_off(buf));
        const float msk = tt[3 * kTile + t];
        float dy[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int c = 0; c < kOut; ++c) {
            const float tg = tt[c * kTile + t];
            const float r = y[c] - tg;
            const float den = y[c] * y[c] + a.loss_eps;
            dy[c] = msk * a.dy_scale * r / den;
            loss += msk * r * r / den;
            jerr += msk * fabsf(r);
            jtgt += msk * fabsf(tg);
        }
        {
            const float zero8[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            store_row8(smem + kSmDY, kDYStride, t, 0u, dy);
            store_row8(smem + kSmDY, kDYStride, t, 8u, zero8);
        }
        sync_operands();
        if (abort_s) break;

        // ---- dH2 = dY W3 (K = 16)
        if (t == 0) {
            tc::fence_after_sync();
            tc::mma_bf16(tmem + kTmD2, tc::smem_desc(sm + kSmDY, 128u, kDYStride),
                         tc::smem_desc(sm + kSmImg + kImgW3PT, 128u, 256u), tc::idesc_bf16(128, 64), 0u);
            commit_mma();
        }
        mma_wait();
        tmem_ld64(tmem, warp, kTmD2, z);
#pragma unroll
        for (int j = 0; j < 64; ++j) z[j] = ((m2[j >> 5] >> (j & 31)) & 1u) ? z[j] : 0.0f;
#pragma unroll
        for (int j = 0; j < 8; ++j) store_row8(smem + kSmZ, kZStride, t, 8u * j, z + 8 * j);
        sync_operands();
        if (abort_s) break;

        // ---- dH1 = dZ2 W2
        if (t == 0) {
            tc::fence_after_sync();
            for (uint32_t ks = 0; ks < kHid / 16; ++ks)
                tc::mma_bf16(tmem + kTmD1, tc::smem_desc(sm + kSmZ + ks * 256u, 128u, kZStride),
                             tc::smem_desc(sm + kSmImg + kImgW2T + ks * 256u, 128u, 1024u), tc::idesc_bf16(128, 64), ks);
            commit_mma();
        }
        mma_wait();
        tmem_ld64(tmem, warp, kTmD1, z);
#pragma unroll
        for (int j = 0; j < 64; ++j) z[j] = ((m1[j >> 5] >> (j & 31)) & 1u) ? z[j] : 0.0f;
#pragma unroll
        for (int j = 0; j < 8; ++j) store_row8(smem + kSmZ, kZStride, t, 64u + 8u * j, z + 8 * j);
        sync_operands();
        if (abort_s) break;

        // ---- dX = dZ1 W1; weight gradients over the tile's samples (MN-major operands):
        //      [dW2 | dW1] += [dZ2 | dZ1]^T [H1 | X],  dW3^T += H2^T dY
        if (t == 0) {
            tc::fence_after_sync();
            for (uint32_t ks = 0; ks < kHid / 16; ++ks)
                tc::mma_bf16(tmem + kTmD1, tc::smem_desc(sm + kSmZ + 1024u + ks * 256u, 128u, kZStride),
                             tc::smem_desc(sm + kSmImg + kImgW1T + ks * 256u, 128u, 1024u), tc::idesc_bf16(128, 32), ks);
            for (uint32_t ks = 0; ks < kTile / 16; ++ks)
                tc::mma_bf16(tmem + kTmGA, tc::smem_desc(sm + kSmZ + ks * 2u * kZStride, kZStride, 128u),
                             tc::smem_desc(xh + ks * 2u * kXHStride, kXHStride, 128u), idesc_mn(128, 96),
                             (it | ks) != 0u);
            // rows 64..127 of this A operand run past H2 into the dY tile: they only feed
            // accumulator rows that are never read
            for (uint32_t ks = 0; ks < kTile / 16; ++ks)
                tc::mma_bf16(tmem + kTmGC, tc::smem_desc(sm + kSmH2 + ks * 2u * kH2Stride, kH2Stride, 128u),
                             tc::smem_desc(sm + kSmDY + ks * 2u * kDYStride, kDYStride, 128u), idesc_mn(128, 16),
                             (it | ks) != 0u);
            commit_mma();
        }
        mma_wait();
        {
            float g0[16], g1[16];
            tc::tmem_ld16(tc::tmem_lane_addr(tmem, warp, kTmD1), g0);
            tc::tmem_ld16(tc::tmem_lane_addr(tmem, warp, kTmD1 + 16), g1);
            tc::wait_ld();
            float4 *dst = reinterpret_cast<float4 *>(a.dX + (size_t)s * kIn);
#pragma unroll
            for (int j = 0; j < 4; ++j) dst[j] = make_float4(g0[4 * j], g0[4 * j + 1], g0[4 * j + 2], g0[4 * j + 3]);
#pragma unroll
            for (int j = 0; j < 4; ++j) dst[4 + j] = make_float4(g1[4 * j], g1[4 * j + 1], g1[4 * j + 2], g1[4 * j + 3]);
        }
        tc::fence_before_sync();
        if (!ok) abort_s = 1;
        __syncthreads();
        if (abort_s) break;
    }

    float *part = a.wpart + (size_t)bid * kPartStride;
    if (abort_s) {
        if (t == 0) {
            atomicOr(a.err, kErrTimeout);
            // what thread 0 started and has not seen complete: the weight image, one load per
            // buffer, one MMA group (a buffer is reloaded, and an MMA group committed, only after
            // the previous one was waited for, so each barrier has at most one phase pending)
            if (!w_done) tc::mbar_wait(&bar_w, 0);
            for (int b = 0; b < 2; ++b)
                if (ld_issued[b] > ld_done[b]) tc::mbar_wait(&bar_ld[b], (ld_issued[b] - 1u) & 1u);
            if (mma_issued > mma_done) tc::mbar_wait(&bar_mma, (mma_issued - 1u) & 1u);
        }
        for (int i = t; i < kPartStride; i += kTile) part[i] = 0.0f;
    } else if (it > 0) {
        // weight gradients of this CTA's tiles: rows 0..63 of GA are dW2, rows 64..127 columns
        // 64..95 are dW1; rows 0..63 of GC are dW3^T.  Plain stores into the CTA's partial row.
        tc::fence_after_sync();
        if (warp < 2) {
            float z[64];
            tmem_ld64(tmem, warp, kTmGA, z);
            float4 *d2 = reinterpret_cast<float4 *>(part + kW2 + t * kHid);
#pragma unroll
            for (int j = 0; j < 16; ++j) d2[j] = make_float4(z[4 * j], z[4 * j + 1], z[4 * j + 2], z[4 * j + 3]);
            float g[16];
            tc::tmem_ld16(tc::tmem_lane_addr(tmem, warp, kTmGC), g);
            tc::wait_ld();
            for (int c = 0; c < kOut; ++c) part[kW3 + c * kHid + t] = g[c];
        } else {
            float g0[16], g1[16];
            tc::tmem_ld16(tc::tmem_lane_addr(tmem, warp, kTmGA + 64), g0);
            tc::tmem_ld16(tc::tmem_lane_addr(tmem, warp, kTmGA + 80), g1);
            tc::wait_ld();
            float4 *d1 = reinterpret_cast<float4 *>(part + kW1 + (t - 64) * kIn);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                d1[j] = make_float4(g0[4 * j], g0[4 * j + 1], g0[4 * j + 2], g0[4 * j + 3]);
                d1[4 + j] = make_float4(g1[4 * j], g1[4 * j + 1], g1[4 * j + 2], g1[4 * j + 3]);
            }
        }
        for (int d = 16; d; d >>= 1) {
            loss += __shfl_xor_sync(0xFFFFFFFFu, loss, d);
            jerr += __shfl_xor_sync(0xFFFFFFFFu, jerr, d);
            jtgt += __shfl_xor_sync(0xFFFFFFFFu, jtgt, d);
        }
        __shared__ float red_s[4][3];
        if ((t & 31) == 0) {
            red_s[warp][0] = loss;
            red_s[warp][1] = jerr;
            red_s[warp][2] = jtgt;
        }
        __syncthreads();
        if (t < 3) part[kWCount + t] = (red_s[0][t] + red_s[1][t] + red_s[2][t] + red_s[3][t]) * (t == 0 ? 0.5f * a.dy_scale : 1.0f);
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, kTmCols);
}

// Forward only, four CTAs of 128 threads per SM (two with the training kernel's layout: 43 us for
// 323 k samples, a chain of three products and three tensor-memory reads per tile with too little
// else on the SM; 25 us with four).  The hidden layers share one shared-memory tile and one
// accumulator: each product has completed before its operand or accumulator is written again.
__global__ void __launch_bounds__(kTile, 4) k_nrc_infer(InferArgs a) {
    const uint32_t bid = blockIdx.x + pass_begin();
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ __align__(8) uint64_t bar_w, bar_ld[2], bar_mma;
    __shared__ uint32_t tmem_s;
    __shared__ int abort_s;
    const uint32_t t = threadIdx.x, warp = t >> 5;
    uint32_t n = a.n;
    if (a.count) n = min(ld(a.count), a.n);
    const uint32_t tiles = (n + kTile - 1) / kTile;
    if (bid >= tiles) return;
    if (t == 0) {
        abort_s = 0;
        tc::mbar_init(&bar_w, 1);
        tc::mbar_init(&bar_ld[0], 1);
        tc::mbar_init(&bar_ld[1], 1);
        tc::mbar_init(&bar_mma, 1);
        tc::mbar_init_fence();
    }
    if (warp == 0) {
        tc::tmem_alloc(&tmem_s, kInfCols);
        tc::tmem_relinquish();
    }
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = tmem_s, sm = tc::smem_u32(smem);
    // what thread 0 started and saw complete (see k_nrc_mlp)
    uint32_t ld_issued[2] = {0u, 0u}, ld_done[2] = {0u, 0u}, mma_issued = 0u, mma_done = 0u;
    auto load_tile = [&](uint32_t tile, int buf) {  // thread 0 only
        ++ld_issued[buf];
        tc::mbar_expect_tx(&bar_ld[buf], kXTile);
        tc::bulk_g2s(smem + kInfX + buf * kXTile, reinterpret_cast<const uint8_t *>(a.X) + (size_t)tile * kXTile, kXTile,
                     &bar_ld[buf]);
    };
    if (t == 0) {
        tc::mbar_expect_tx(&bar_w, kInfX);
        tc::bulk_g2s(smem + kInfW1, a.wimg + kImgW1, kInfW2 - kInfW1, &bar_w);
        tc::bulk_g2s(smem + kInfW2, a.wimg + kImgW2, kInfW3 - kInfW2, &bar_w);
        tc::bulk_g2s(smem + kInfW3, a.wimg + kImgW3P, kInfX - kInfW3, &bar_w);
        load_tile(bid, 0);
    }
    const bool w_done = tc::mbar_wait(&bar_w, 0);
    bool ok = w_done;
    uint32_t ph = 0, it = 0;
    auto commit_mma = [&]() {  // thread 0 only
        tc::commit(&bar_mma);
        ++mma_issued;
    };
    auto mma_wait = [&]() {
        const bool got = tc::mbar_wait(&bar_mma, ph);
        if (got) ++mma_done;
        ok = got && ok;
        ph ^= 1u;
        tc::fence_after_sync();
    };
    // this thread's row of a hidden layer: ReLU, bf16, into the shared tile; then every row is there
    auto hidden = [&]() {
        float z[64];
        tmem_ld64(tmem, warp, kInfD, z);
#pragma unroll
        for (int j = 0; j < 64; ++j) z[j] = fmaxf(z[j], 0.0f);
#pragma unroll
        for (int j = 0; j < 8; ++j) store_row8(smem + kInfH, kH2Stride, t, 8u * j, z + 8 * j);
        tc::fence_async_smem();
        tc::fence_before_sync();
        if (!ok) abort_s = 1;
        __syncthreads();
    };
    for (uint32_t tile = bid; tile < tiles; tile += gridDim.x, ++it) {
        const int buf = it & 1;
        const bool got = tc::mbar_wait(&bar_ld[buf], (it >> 1) & 1u);
        if (got) ++ld_done[buf];
        ok = got && ok;
        if (!ok) abort_s = 1;
        tc::fence_before_sync();
        __syncthreads();  // the previous tile's output has been read out of tensor memory
        if (abort_s) break;
        if (t == 0) {
            if (tile + gridDim.x < tiles) load_tile(tile + gridDim.x, buf ^ 1);
            tc::fence_after_sync();
            for (uint32_t ks = 0; ks < kIn / 16; ++ks)
                tc::mma_bf16(tmem + kInfD, tc::smem_desc(sm + kInfX + buf * kXTile + ks * 256u, 128u, 512u),
                             tc::smem_desc(sm + kInfW1 + ks * 256u, 128u, 512u), tc::idesc_bf16(128, 64), ks);
            commit_mma();
        }
        mma_wait();
        hidden();
        if (abort_s) break;
        if (t == 0) {
            tc::fence_after_sync();
            for (uint32_t ks = 0; ks < kHid / 16; ++ks)
                tc::mma_bf16(tmem + kInfD, tc::smem_desc(sm + kInfH + ks * 256u, 128u, kH2Stride),
                             tc::smem_desc(sm + kInfW2 + ks * 256u, 128u, 1024u), tc::idesc_bf16(128, 64), ks);
            commit_mma();
        }
        mma_wait();
        hidden();
        if (abort_s) break;
        if (t == 0) {
            tc::fence_after_sync();
            for (uint32_t ks = 0; ks < kHid / 16; ++ks)
                tc::mma_bf16(tmem + kInfD3, tc::smem_desc(sm + kInfH + ks * 256u, 128u, kH2Stride),
                             tc::smem_desc(sm + kInfW3 + ks * 256u, 128u, 1024u), tc::idesc_bf16(128, 16), ks);
            commit_mma();
        }
        mma_wait();
        float y[16];
        tc::tmem_ld16(tc::tmem_lane_addr(tmem, warp, kInfD3), y);
        tc::wait_ld();
        const uint32_t s = tile * kTile + t;
        if (s < n && ok) {
            const uint32_t o = a.out_idx ? __ldca(a.out_idx + s) : s;
            a.out[o] = make_float4(fmaxf(y[0], 0.0f), fmaxf(y[1], 0.0f), fmaxf(y[2], 0.0f), 1.0f);
        }
    }
    if (!ok) abort_s = 1;
    tc::fence_before_sync();
    __syncthreads();
    if (abort_s && t == 0) {
        atomicOr(a.err, kErrTimeout);
        if (!w_done) tc::mbar_wait(&bar_w, 0);
        for (int b = 0; b < 2; ++b)
            if (ld_issued[b] > ld_done[b]) tc::mbar_wait(&bar_ld[b], (ld_issued[b] - 1u) & 1u);
        if (mma_issued > mma_done) tc::mbar_wait(&bar_mma, (mma_issued - 1u) & 1u);
    }
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, kInfCols);
}

// ---------------------------------------------------------------- gradient scatter and Adam

// Sum of the network kernel's per-CTA partials of value i (a weight gradient, then the loss sums): a
// block takes 32 consecutive values x 8 warps; warp w sums parts w, w + 8, ...; then the 8 warp sums in
// a fixed order (deterministic).  Warp 0 gets the sum; acc: 8 x 32 floats of shared memory.
__device__ __forceinline__ float wgrad_sum(const float *wpart, int parts, int i, int lane, int w, float *acc) {
    float s = 0.0f;
    if (i < kWCount + 3) {
#pragma unroll 4
        for (int p = w; p < parts; p += 8) s += __ldcg(wpart + (size_t)p * kPartStride + i);
    }
    acc[32 * w + lane] = s;
    __syncthreads();
    float t = 0.0f;
    if (w == 0) {
#pragma unroll
        for (int k = 0; k < 8; ++k) t += acc[32 * k + lane];
    }
    return t;
}

// ... added to the weight-gradient accumulators and the loss sums.
__global__ void __launch_bounds__(256) k_nrc_wgrad_reduce(const float *wpart, int parts, float *wg, float *stats) {
    const uint32_t bid = blockIdx.x + pass_begin();
    __shared__ float acc[8 * 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int i = bid * 32 + lane;
    const float t = wgrad_sum(wpart, parts, i, lane, w, acc);
    if (w == 0 && i < kWCount + 3) {
        if (i < kWCount) wg[i] += t;
        else stats[i - kWCount] += t;
    }
}

__global__ void __launch_bounds__(kEncThreads) k_nrc_scatter(ScatterArgs a) {
    const uint32_t bid = blockIdx.x + pass_begin();
    const uint32_t T = 1u << a.geo.log2_table;
    for (uint32_t i = bid * blockDim.x + threadIdx.x; i < a.n * kL; i += gridDim.x * blockDim.x) {
        const uint32_t s = i >> 4, l = i & 15u;
        const float2 g = __ldca(reinterpret_cast<const float2 *>(a.dX + (size_t)s * kIn) + l);
        if (g.x == 0.0f && g.y == 0.0f) continue;
        const uint32_t r = a.idx ? __ldca(a.idx + s) : s;
        float x[3];
        normalise(a.geo, __ldca(a.pos[0] + r), __ldca(a.pos[1] + r), __ldca(a.pos[2] + r), x);
        const uint32_t d = dir_code(__ldca(a.nrm[0] + r), __ldca(a.nrm[1] + r), __ldca(a.nrm[2] + r));
        uint32_t idx[8];
        float w[8];
        level_corners(x, a.geo.lv.res[l], a.geo.lv.dense[l] != 0u, d, T - 1u, idx, w);
        float2 *gt = a.grad + (size_t)l * T;
#pragma unroll
        for (int c = 0; c < 8; ++c) atomicAdd(gt + idx[c], make_float2(w[c] * g.x, w[c] * g.y));
    }
}

struct AdamArgs {
    float lr, b1, b2, eps, c1, c2;  // c1 = 1 - b1^t, c2 = 1 - b2^t
};

__device__ __forceinline__ float adam_update(float p, float &m, float &v, float g, const AdamArgs &a) {
    m = a.b1 * m + (1.0f - a.b1) * g;
    v = a.b2 * v + (1.0f - a.b2) * g * g;
    return p - a.lr * (m / a.c1) / (sqrtf(v / a.c2) + a.eps);
}

struct AdamTableArgs {
    Entry *tab;
    float2 *grad;
    __half2 *tab16;
    uint32_t log2_table;
    uint32_t chunk0[kL + 1];  // first chunk of entries of each level, then their number
};
constexpr int kAdamWarps = 8, kAdamBlocksPerSm = 4;

// Sparse Adam on the table: an entry whose gradient is (0, 0) this step keeps its value and its
// moments (the samples of the step did not touch it); the others take an Adam step with the
// global step count's bias correction.  Gradients are cleared as they are consumed.
// A step touches an eighth of the entries, at hash-random places.  A warp therefore reads the
// gradients of 256 consecutive entries (four 16-byte loads a lane in flight), lists the touched ones in
// shared memory and updates the list lane by lane, so that every lane holds an entry's loads and
// arithmetic instead of one in eight (4 entries a thread, skipping the untouched: 40 us a step of 16,384
// samples, 2^19 entries a level; this form with the weights 27.5 us).  Where that leaves resident warps
// without a chunk, a warp takes 64 entries: small tables are touched all over, and a warp's 256 follow one
// another in four trips (10,000 samples, 2^14 entries a level, backward and step: 47 us with 256, 34.5 with 64).
template <int CHUNK>
__device__ __forceinline__ void adam_table(const AdamTableArgs &t, const AdamArgs &a, uint32_t warp, uint32_t warps,
                                           float2 *s_g, uint16_t *s_i) {
    const uint32_t lane = threadIdx.x & 31u;
    for (uint32_t c = warp; c < t.chunk0[kL]; c += warps) {
        uint32_t l = 0;
#pragma unroll
        for (int k = 1; k < kL; ++k) l += c >= t.chunk0[k] ? 1u : 0u;
        uint32_t first = t.chunk0[0];
#pragma unroll
        for (int k = 1; k < kL; ++k) first = c >= t.chunk0[k] ? t.chunk0[k] : first;
        const size_t e0 = ((size_t)l << t.log2_table) + (size_t)(c - first) * CHUNK;
        float4 *gq = reinterpret_cast<float4 *>(t.grad + e0);
        float4 g[CHUNK / 64];
#pragma unroll
        for (int j = 0; j < CHUNK / 64; ++j) g[j] = __ldcg(gq + 32 * j + lane);
        uint32_t hit = 0;
#pragma unroll
        for (int j = 0; j < CHUNK / 64; ++j) {
            if (g[j].x != 0.0f || g[j].y != 0.0f) hit |= 1u << (2 * j);
            if (g[j].z != 0.0f || g[j].w != 0.0f) hit |= 2u << (2 * j);
            if ((hit >> (2 * j)) & 3u) gq[32 * j + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        const int cnt = __popc(hit);
        int incl = cnt;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int v = __shfl_up_sync(0xFFFFFFFFu, incl, d);
            if ((int)lane >= d) incl += v;
        }
        const int total = __shfl_sync(0xFFFFFFFFu, incl, 31);
        int pos = incl - cnt;
#pragma unroll
        for (int j = 0; j < CHUNK / 64; ++j) {
            if ((hit >> (2 * j)) & 1u) {
                s_i[pos] = (uint16_t)(64 * j + 2 * lane);
                s_g[pos++] = make_float2(g[j].x, g[j].y);
            }
            if ((hit >> (2 * j)) & 2u) {
                s_i[pos] = (uint16_t)(64 * j + 2 * lane + 1);
                s_g[pos++] = make_float2(g[j].z, g[j].w);
            }
        }
        __syncwarp();
        for (int k = (int)lane; k < total; k += 64) {
            float4 pm[2], vp[2];
            size_t e[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                if (k + 32 * u >= total) continue;
                e[u] = e0 + s_i[k + 32 * u];
                const float4 *src = reinterpret_cast<const float4 *>(t.tab + e[u]);
                pm[u] = __ldcg(src);
                vp[u] = __ldcg(src + 1);
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                if (k + 32 * u >= total) continue;
                const float2 gr = s_g[k + 32 * u];
                pm[u].x = adam_update(pm[u].x, pm[u].z, vp[u].x, gr.x, a);
                pm[u].y = adam_update(pm[u].y, pm[u].w, vp[u].y, gr.y, a);
                float4 *dst = reinterpret_cast<float4 *>(t.tab + e[u]);
                dst[0] = pm[u];
                dst[1] = vp[u];
                t.tab16[e[u]] = __floats2half2_rn(pm[u].x, pm[u].y);
            }
        }
        __syncwarp();
    }
}

__global__ void k_nrc_table_f16(const Entry *tab, __half2 *tab16, uint64_t n) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
        tab16[i] = __floats2half2_rn(tab[i].p.x, tab[i].p.y);
}

// Master features <-> a plain float2 array: mode 0 reads them out, 1 writes them, 2 clears the
// Adam moments (buf unused).
__global__ void k_nrc_table_field(Entry *tab, float2 *buf, uint64_t n, int mode) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        if (mode == 2) tab[i].m = tab[i].v = make_float2(0.0f, 0.0f);
        else if (mode == 1) tab[i].p = buf[i];
        else buf[i] = tab[i].p;
    }
}

__device__ __forceinline__ void put_bf16(uint8_t *img, uint32_t off, float v) {
    *reinterpret_cast<__nv_bfloat16 *>(img + off) = __float2bfloat16_rn(v);
}

// Weight i's value into the bf16 images W, W^T of its layer.
__device__ __forceinline__ void weight_images(uint8_t *img, int i, float p) {
    if (i < kW2) {
        const uint32_t o = i / kIn, k = i % kIn;
        put_bf16(img, kImgW1 + tc::cm_offset(o, k, kIn), p);
        put_bf16(img, kImgW1T + tc::cm_offset(k, o, kHid), p);
    } else if (i < kW3) {
        const uint32_t o = (i - kW2) / kHid, k = (i - kW2) % kHid;
        put_bf16(img, kImgW2 + tc::cm_offset(o, k, kHid), p);
        put_bf16(img, kImgW2T + tc::cm_offset(k, o, kHid), p);
    } else {
        const uint32_t o = (i - kW3) / kHid, k = (i - kW3) % kHid;
        put_bf16(img, kImgW3P + tc::cm_offset(o, k, kHid), p);
        put_bf16(img, kImgW3PT + tc::cm_offset(k, o, 16), p);
    }
}

// The bf16 images from the master weights.
__global__ void __launch_bounds__(256) k_nrc_images(const float *w, uint8_t *img) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < kWCount) weight_images(img, i, w[i]);
}

// One Adam step: blocks 0 .. kAdamWBlocks - 1 take 32 weights (and the loss sums) each, with the
// network kernel's per-CTA partials added to their gradients as k_nrc_wgrad_reduce does (parts = 0:
// none), the others the table.  One launch, so that the weights' two short passes cost no launches of
// their own (4.9 and 2.9 us a step).
struct AdamWeightArgs {
    float *w, *m, *v, *g;
    uint8_t *img;
    const float *wpart;
    int parts;
    float *stats;
};
constexpr int kAdamWBlocks = (kWCount + 3 + 31) / 32;
template <int CHUNK>
__global__ void __launch_bounds__(32 * kAdamWarps, kAdamBlocksPerSm) k_nrc_adam(AdamTableArgs t, AdamWeightArgs q, AdamArgs a) {
    const uint32_t bid = blockIdx.x + pass_begin();
    __shared__ float2 s_g[kAdamWarps][CHUNK];
    __shared__ uint16_t s_i[kAdamWarps][CHUNK];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (bid >= kAdamWBlocks) {
        adam_table<CHUNK>(t, a, (bid - kAdamWBlocks) * kAdamWarps + w, (gridDim.x - kAdamWBlocks) * kAdamWarps, s_g[w],
                   s_i[w]);
        return;
    }
    const int i = bid * 32 + lane;
    const float sum = wgrad_sum(q.wpart, q.parts, i, lane, w, &s_g[0][0].x);
    if (w != 0 || i >= kWCount + 3) return;
    if (i >= kWCount) {
        if (q.parts) q.stats[i - kWCount] += sum;
        return;
    }
    float mm = q.m[i], vv = q.v[i];
    const float g = q.parts ? q.g[i] + sum : q.g[i];
    const float p = adam_update(q.w[i], mm, vv, g, a);
    q.m[i] = mm;
    q.v[i] = vv;
    q.g[i] = 0.0f;
    q.w[i] = p;
    weight_images(q.img, i, p);
}

// ---------------------------------------------------------------- query selection

// A block takes 32 words (1024 records) at a time: each warp decides its 2 words, the block's answered
// records take consecutive places with one addition to the counter (one addition per warp of 32
// records, 64,800 at 1080p on one address, took 57 us).  What bounds a round is its chain of
// dependent loads, so a warp reads the planes and slots of its words in one trip and the cells' cold
// marks in a second: 17 us at 1080p and 5.1 us for 230,400 records, against 30 and 24 us word after word.
constexpr int kSelWarps = 16, kSelWords = 2;
__global__ void __launch_bounds__(32 * kSelWarps) k_nrc_select(SelectArgs a) {
    const uint32_t bid = blockIdx.x + pass_begin();
    __shared__ uint32_t s_cnt[kSelWarps], s_base;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const bool trusted = a.trained && ld(a.stats + 2) > 0.0f && ld(a.stats + 1) <= a.trust * ld(a.stats + 2);
    const uint32_t words = (a.n + 31u) / 32u;
    for (uint32_t b0 = bid * (kSelWarps * kSelWords); b0 < words; b0 += gridDim.x * (kSelWarps * kSelWords)) {
        const uint32_t w0 = b0 + warp * kSelWords;
        float len[kSelWords], px[kSelWords], py[kSelWords], pz[kSelWords];
        uint32_t slot[kSelWords], ball[kSelWords], total = 0;
#pragma unroll
        for (int k = 0; k < kSelWords; ++k) {
            const uint32_t r = (w0 + k) * 32u + lane;
            len[k] = -1.0f;
            px[k] = py[k] = pz[k] = 0.0f;
            slot[k] = GI_SLOT_MISS;
            if (r < a.n) {
                len[k] = __ldca(a.len + r);
                px[k] = __ldca(a.pos[0] + r);
                py[k] = __ldca(a.pos[1] + r);
                pz[k] = __ldca(a.pos[2] + r);
                slot[k] = __ldca(a.slot_ids + r);
            }
        }
        bool use[kSelWords];
#pragma unroll
        for (int k = 0; k < kSelWords; ++k) {
            const bool hit = isfinite(len[k]) && len[k] >= 0.0f && isfinite(px[k]) && isfinite(py[k]) && isfinite(pz[k]);
            // GI_SLOT_FAR: left out of the table by the update (gi_cache_route_far), the network is its only answer
            use[k] = hit && (slot[k] == GI_SLOT_FAR || (trusted && slot[k] == GI_SLOT_NONE));
            if (hit && trusted && slot[k] < a.cv.slots)
                use[k] = cache_cold(a.cv, slot[k]) || key_lod(a.kp, px[k], py[k], pz[k]) >= (int)a.query_lod;
        }
#pragma unroll
        for (int k = 0; k < kSelWords; ++k) {
            ball[k] = __ballot_sync(0xFFFFFFFFu, use[k]);
            total += __popc(ball[k]);
        }
        if (lane == 0) s_cnt[warp] = total;
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t sum = 0;
            for (int w = 0; w < kSelWarps; ++w) {
                const uint32_t c = s_cnt[w];
                s_cnt[w] = sum;
                sum += c;
            }
            s_base = sum ? atomicAdd(a.qcount, sum) : 0u;
        }
        __syncthreads();
        uint32_t base = s_base + s_cnt[warp];
#pragma unroll
        for (int k = 0; k < kSelWords; ++k) {
            const uint32_t pos = base + __popc(ball[k] & ((1u << lane) - 1u));
            const bool take = ((ball[k] >> lane) & 1u) && pos < a.max_q;
            if (take) a.qidx[pos] = (w0 + k) * 32u + lane;
            const uint32_t kept = __ballot_sync(0xFFFFFFFFu, take);
            if (lane == 0 && w0 + k < words) a.bits[w0 + k] = kept;
            base += __popc(ball[k]);
        }
        __syncthreads();  // the next round reuses the block's counters
    }
}

__global__ void k_nrc_gather_answers(const uint32_t *qidx, const float4 *ovr, uint32_t count, uint32_t *records,
                                     float4 *rad) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
        const uint32_t r = qidx[i];
        records[i] = r;
        rad[i] = ovr[r];
    }
}

// ---------------------------------------------------------------- host side

uint64_t splitmix64(uint64_t &s) {
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

double uniform01(uint64_t &s) { return (double)(splitmix64(s) >> 11) * (1.0 / 9007199254740992.0); }

int sm_count() {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 1;
}

}  // namespace
}  // namespace gi

struct gi_nrc_s {
    gi_nrc_config cfg;
    gi::Geometry geo;
    uint32_t T;
    gi::Entry *tab = nullptr;
    float2 *grad = nullptr;     // table gradient accumulators [levels][T]
    __half2 *tab16 = nullptr;
    float *w = nullptr, *wm = nullptr, *wv = nullptr, *wg = nullptr;
    uint8_t *wimg = nullptr;
    float *stats = nullptr;      // loss, sum m|y - t|, sum m|t|, spare
    float *wpart = nullptr;      // per-CTA partial weight gradients of the training network kernel
    uint32_t *err = nullptr;
    // per-batch scratch, capacity `cap` samples (a multiple of 128)
    uint32_t cap = 0;
    uint16_t *X = nullptr;
    float *Tt = nullptr;
    float *dX = nullptr;
    uint32_t *idx = nullptr;
    // query state
    uint32_t *bits = nullptr;
    float4 *ovr = nullptr;
    uint32_t *qidx = nullptr;
    uint32_t *qcount = nullptr;
    uint64_t last_query_n = 0;
    bool queried = false;
    uint64_t steps = 0;
    bool grads_set = false;      // table gradients written by the caller since the last Adam step
    uint32_t last_minibatches = 1;
    int sms = 1;
};

using namespace gi;

namespace {

gi_status nrc_alloc(void **p, size_t bytes) {
    if (cudaMalloc(p, bytes) != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        set_error("gi_nrc: cudaMalloc of %zu bytes failed", bytes);
        return GI_ERR_OOM;
    }
    return GI_OK;
}

void nrc_free(gi_nrc_s *s) {
    void *ptrs[] = {s->tab, s->grad, s->tab16, s->w, s->wm, s->wv, s->wg, s->wimg, s->stats, s->err, s->wpart,
                    s->X, s->Tt, s->dX, s->idx, s->bits, s->ovr, s->qidx, s->qcount};
    for (void *p : ptrs)
        if (p) cudaFree(p);
}

gi_status ensure_capacity(gi_nrc_s *s, uint32_t n) {
    const uint32_t need = (n + kTile - 1) / kTile * kTile;
    if (need <= s->cap) return GI_OK;
    cudaDeviceSynchronize();
    for (void *p : {(void *)s->X, (void *)s->Tt, (void *)s->dX, (void *)s->idx})
        if (p) cudaFree(p);
    s->X = nullptr;
    s->Tt = nullptr;
    s->dX = nullptr;
    s->idx = nullptr;
    s->cap = 0;
    gi_status st = nrc_alloc((void **)&s->X, (size_t)need * kIn * 2);
    if (st == GI_OK) st = nrc_alloc((void **)&s->Tt, (size_t)need / kTile * kTTile);
    if (st == GI_OK) st = nrc_alloc((void **)&s->dX, (size_t)need * kIn * 4);
    if (st == GI_OK) st = nrc_alloc((void **)&s->idx, (size_t)need * 4);
    if (st == GI_OK) s->cap = need;
    return st;
}

bool points_ok(const gi_points *p) {
    if (!p || p->n > GI_NRC_MAX_BATCH) return false;
    if (p->n == 0) return true;
    for (int a = 0; a < 3; ++a)
        if (!p->pos[a] || !p->nrm[a]) return false;
    return true;
}

EncArgs enc_base(const gi_nrc_s *s) {
    EncArgs e;
    memset(&e, 0, sizeof(e));
    e.geo = s->geo;
    e.tab16 = s->tab16;
    e.X = s->X;
    e.T = s->Tt;
    e.idx = s->idx;
    return e;
}

// Blocks of the kernels with one thread per sample and level (n samples, padded to whole tiles).
unsigned sample_blocks(const gi_nrc_s *s, uint32_t n) {
    const uint64_t b = (uint64_t)((n + kTile - 1) / kTile * kTile) * kL / kEncThreads;
    return (unsigned)std::min<uint64_t>(b, (uint64_t)s->sms * 8);
}

// The network on n encoded samples, training: *parts rows of partial sums in s->wpart.
gi_status launch_train(gi_nrc_s *s, uint32_t n, float dy_scale, int *parts, cudaStream_t st) {
    MlpArgs m;
    m.X = s->X;
    m.T = s->Tt;
    m.wimg = s->wimg;
    m.n = n;
    m.dy_scale = dy_scale;
    m.loss_eps = s->cfg.loss_eps;
    m.dX = s->dX;
    m.wpart = s->wpart;
    m.err = s->err;
    const uint32_t tiles = (n + kTile - 1) / kTile;
    *parts = (int)std::min<uint32_t>(tiles, (uint32_t)s->sms);
    if (tiles == 0) return GI_OK;
    launch(k_nrc_mlp, *parts, kTile, kSmTrain, st, m);
    return cuda_status(cudaGetLastError(), "k_nrc_mlp launch");
}

// Forward only; count: device sample count (at most n), or NULL.
gi_status launch_infer(gi_nrc_s *s, uint32_t n, const uint32_t *count, float4 *out, const uint32_t *out_idx,
                       cudaStream_t st) {
    const uint32_t tiles = (n + kTile - 1) / kTile;
    if (tiles == 0) return GI_OK;
    const InferArgs m = {s->X, s->wimg, n, count, out, out_idx, s->err};
    launch(k_nrc_infer, std::min<uint32_t>(tiles, 4u * (uint32_t)s->sms), kTile, kInfBytes, st, m);
    return cuda_status(cudaGetLastError(), "k_nrc_infer launch");
}

gi_status scatter_and_return(gi_nrc_s *s, const float *const pos[3], const float *const nrm[3], const uint32_t *idx,
                             uint32_t n, cudaStream_t st) {
    ScatterArgs c;
    c.geo = s->geo;
    for (int a = 0; a < 3; ++a) {
        c.pos[a] = pos[a];
        c.nrm[a] = nrm[a];
    }
    c.idx = idx;
    c.n = n;
    c.dX = s->dX;
    c.grad = s->grad;
    launch(k_nrc_scatter, sample_blocks(s, n), kEncThreads, 0, st, c);
    return cuda_status(cudaGetLastError(), "k_nrc_scatter launch");
}

gi_status table_field(gi_nrc_s *s, float2 *host, bool grads, int mode) {
    const uint64_t entries = (uint64_t)kL * s->T;
    cudaError_t e = cudaSuccess;
    if (grads) {  // the gradient array is a plain float2 array already
        if (mode == 1) e = cudaMemcpy(s->grad, host, entries * sizeof(float2), cudaMemcpyHostToDevice);
        else e = cudaMemcpy(host, s->grad, entries * sizeof(float2), cudaMemcpyDeviceToHost);
        return cuda_status(e, "gi_nrc gradient transfer");
    }
    const unsigned blocks = (unsigned)std::min<uint64_t>((entries + 255) / 256, 65535);
    float2 *tmp = nullptr;
    if (mode != 2) {
        gi_status st = nrc_alloc((void **)&tmp, entries * sizeof(float2));
        if (st != GI_OK) return st;
    }
    if (mode == 1) e = cudaMemcpy(tmp, host, entries * sizeof(float2), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        k_nrc_table_field<<<blocks, 256>>>(s->tab, tmp, entries, mode);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e == cudaSuccess && mode == 0) e = cudaMemcpy(host, tmp, entries * sizeof(float2), cudaMemcpyDeviceToHost);
    if (tmp) cudaFree(tmp);
    return cuda_status(e, "gi_nrc table transfer");
}

gi_status copy_params(gi_nrc_s *s, const float *table, const float *w1, const float *w2, const float *w3, bool grads) {
    gi_status st = GI_OK;
    if (table) st = table_field(s, reinterpret_cast<float2 *>(const_cast<float *>(table)), grads, 1);
    float *dst = grads ? s->wg : s->w;
    cudaError_t e = cudaSuccess;
    if (st == GI_OK && w1) e = cudaMemcpy(dst + kW1, w1, sizeof(float) * kHid * kIn, cudaMemcpyHostToDevice);
    if (e == cudaSuccess && st == GI_OK && w2) e = cudaMemcpy(dst + kW2, w2, sizeof(float) * kHid * kHid, cudaMemcpyHostToDevice);
    if (e == cudaSuccess && st == GI_OK && w3) e = cudaMemcpy(dst + kW3, w3, sizeof(float) * kOut * kHid, cudaMemcpyHostToDevice);
    return st != GI_OK ? st : cuda_status(e, "gi_nrc parameter upload");
}

gi_status read_params(gi_nrc_s *s, float *table, float *w1, float *w2, float *w3, bool grads) {
    gi_status st = cuda_status(cudaDeviceSynchronize(), "gi_nrc parameter download");
    if (st == GI_OK && table) st = table_field(s, reinterpret_cast<float2 *>(table), grads, 0);
    const float *src = grads ? s->wg : s->w;
    cudaError_t e = cudaSuccess;
    if (st == GI_OK && w1) e = cudaMemcpy(w1, src + kW1, sizeof(float) * kHid * kIn, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess && st == GI_OK && w2) e = cudaMemcpy(w2, src + kW2, sizeof(float) * kHid * kHid, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess && st == GI_OK && w3) e = cudaMemcpy(w3, src + kW3, sizeof(float) * kOut * kHid, cudaMemcpyDeviceToHost);
    return st != GI_OK ? st : cuda_status(e, "gi_nrc parameter download");
}

// refresh the float16 table copy and the bf16 weight images from the masters (no Adam step)
gi_status refresh_copies(gi_nrc_s *s) {
    const uint64_t entries = (uint64_t)kL * s->T;
    k_nrc_table_f16<<<(unsigned)std::min<uint64_t>((entries + 255) / 256, 65535), 256>>>(s->tab, s->tab16, entries);
    k_nrc_images<<<(kWCount + 255) / 256, 256>>>(s->w, s->wimg);
    gi_status st = cuda_status(cudaGetLastError(), "gi_nrc copy refresh");
    if (st == GI_OK) st = cuda_status(cudaDeviceSynchronize(), "gi_nrc copy refresh");
    return st;
}

}  // namespace

namespace gi {
void nrc_route_inputs(gi_nrc_t nrc, const float **stats, float *trust, bool *trained) {
    *stats = nrc->stats;
    *trust = nrc->cfg.trust;
    *trained = nrc->steps > 0;
}

gi_status nrc_override(gi_nrc_t nrc, uint64_t n, const uint32_t **bits, const float4 **ovr) {
    if (!nrc->queried || nrc->last_query_n != n) {
        set_error("gi_probes_integrate_nrc: no gi_nrc_query_frame for a view of %llu records", (unsigned long long)n);
        return GI_ERR_INVALID_ARG;
    }
    *bits = nrc->bits;
    *ovr = nrc->ovr;
    return GI_OK;
}
}  // namespace gi

extern "C" {

gi_status gi_nrc_config_defaults(gi_nrc_config *cfg) {
    if (!cfg) {
        set_error("gi_nrc_config_defaults: NULL config");
        return GI_ERR_INVALID_ARG;
    }
    memset(cfg, 0, sizeof *cfg);
    cfg->log2_table = 19;
    // geometric level schedule from 16 to 2048 cells per axis (Mueller et al. 2022, Section 3)
    const double n_min = 16.0, n_max = 2048.0;
    const double b = pow(n_max / n_min, 1.0 / (GI_NRC_LEVELS - 1));
    for (int l = 0; l < GI_NRC_LEVELS; ++l) cfg->resolution[l] = (uint32_t)floor(n_min * pow(b, (double)l) + 1e-9);
    cfg->resolution[GI_NRC_LEVELS - 1] = (uint32_t)n_max;
    for (int a = 0; a < 3; ++a) {
        cfg->aabb_lo[a] = 0.0f;
        cfg->aabb_hi[a] = 1.0f;
    }
    cfg->lr = 1e-2f;
    cfg->beta1 = 0.9f;
    cfg->beta2 = 0.99f;
    cfg->adam_eps = 1e-15f;
    cfg->loss_eps = 0.01f;
    cfg->batch = 65536;
    cfg->train_steps = 4;
    cfg->max_records = 1u << 22;
    cfg->max_queries = 1u << 20;
    cfg->trust = 0.05f;
    cfg->query_lod = 2;
    cfg->seed = 1;
    return GI_OK;
}

gi_status gi_nrc_create(const gi_nrc_config *cfg, gi_nrc_t *out) {
    if (!cfg || !out) {
        set_error("gi_nrc_create: NULL argument");
        return GI_ERR_INVALID_ARG;
    }
    *out = nullptr;
    bool ok = cfg->log2_table >= 10 && cfg->log2_table <= 24 && cfg->lr > 0.f && cfg->beta1 >= 0.f &&
              cfg->beta1 < 1.f && cfg->beta2 >= 0.f && cfg->beta2 < 1.f && cfg->adam_eps >= 0.f &&
              cfg->loss_eps > 0.f && cfg->batch >= 128 && cfg->batch <= GI_NRC_MAX_BATCH && cfg->train_steps >= 1 &&
              cfg->batch % cfg->train_steps == 0 && cfg->batch / cfg->train_steps >= 128 && cfg->trust >= 0.f &&
              cfg->max_queries <= GI_NRC_MAX_BATCH;
    for (int l = 0; l < kL; ++l) ok = ok && cfg->resolution[l] >= 1 && cfg->resolution[l] <= (1u << 20);
    for (int a = 0; a < 3; ++a) ok = ok && std::isfinite(cfg->aabb_lo[a]) && std::isfinite(cfg->aabb_hi[a]) &&
                                     cfg->aabb_hi[a] > cfg->aabb_lo[a];
    if (!ok) {
        set_error("gi_nrc_create: configuration out of range");
        return GI_ERR_INVALID_ARG;
    }
    gi_nrc_s *s = new gi_nrc_s();
    s->cfg = *cfg;
    s->T = 1u << cfg->log2_table;
    s->sms = sm_count();
    for (int a = 0; a < 3; ++a) {
        s->geo.lo[a] = cfg->aabb_lo[a];
        s->geo.inv_ext[a] = (float)(1.0 / ((double)cfg->aabb_hi[a] - (double)cfg->aabb_lo[a]));
    }
    s->geo.log2_table = cfg->log2_table;
    for (int l = 0; l < kL; ++l) {
        const uint64_t V = (uint64_t)cfg->resolution[l] + 1u;
        s->geo.lv.res[l] = cfg->resolution[l];
        s->geo.lv.dense[l] = 6u * V * V * V <= s->T ? 1u : 0u;
    }
    const size_t entries = (size_t)kL * s->T;
    gi_status st = nrc_alloc((void **)&s->tab, entries * sizeof(Entry));
    if (st == GI_OK) st = nrc_alloc((void **)&s->grad, entries * sizeof(float2));
    if (st == GI_OK) st = nrc_alloc((void **)&s->tab16, entries * sizeof(__half2));
    if (st == GI_OK) st = nrc_alloc((void **)&s->w, kWCount * 4);
    if (st == GI_OK) st = nrc_alloc((void **)&s->wm, kWCount * 4);
    if (st == GI_OK) st = nrc_alloc((void **)&s->wv, kWCount * 4);
    if (st == GI_OK) st = nrc_alloc((void **)&s->wg, kWCount * 4);
    if (st == GI_OK) st = nrc_alloc((void **)&s->wimg, kImgBytes);
    if (st == GI_OK) st = nrc_alloc((void **)&s->stats, 16);
    if (st == GI_OK) st = nrc_alloc((void **)&s->wpart, (size_t)s->sms * kPartStride * 4);
    if (st == GI_OK) st = nrc_alloc((void **)&s->err, 4);
    if (st == GI_OK) st = nrc_alloc((void **)&s->qcount, 4);
    const uint32_t maxr = std::max<uint32_t>(cfg->max_records, 32);
    if (st == GI_OK) st = nrc_alloc((void **)&s->bits, ((size_t)maxr + 31) / 32 * 4 + 8);
    if (st == GI_OK) st = nrc_alloc((void **)&s->ovr, (size_t)maxr * sizeof(float4));
    if (st == GI_OK) st = nrc_alloc((void **)&s->qidx, (size_t)std::max<uint32_t>(cfg->max_queries, 1) * 4);
    if (st == GI_OK) st = ensure_capacity(s, std::max(cfg->batch, cfg->max_queries));
    if (st != GI_OK) {
        nrc_free(s);
        delete s;
        return st;
    }
    cudaError_t e = cudaMemset(s->tab, 0, entries * sizeof(Entry));
    if (e == cudaSuccess) e = cudaMemset(s->grad, 0, entries * sizeof(float2));
    if (e == cudaSuccess) e = cudaMemset(s->wm, 0, kWCount * 4);
    if (e == cudaSuccess) e = cudaMemset(s->wv, 0, kWCount * 4);
    if (e == cudaSuccess) e = cudaMemset(s->wg, 0, kWCount * 4);
    if (e == cudaSuccess) e = cudaMemset(s->wimg, 0, kImgBytes);
    if (e == cudaSuccess) e = cudaMemset(s->stats, 0, 16);
    if (e == cudaSuccess) e = cudaMemset(s->err, 0, 4);
    if (e == cudaSuccess) e = cudaMemset(s->qcount, 0, 4);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_nrc_mlp, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmTrain);
    st = cuda_status(e, "gi_nrc_create");
    if (st == GI_OK) {
        // initial parameters from a splitmix64 stream: table, then W1, W2, W3
        uint64_t rs = cfg->seed;
        std::vector<float> table(entries * 2);
        for (auto &v : table) v = (float)(uniform01(rs) * 2e-4 - 1e-4);
        std::vector<float> w(kWCount);
        const double b1 = std::sqrt(6.0 / (kIn + kHid)), b2 = std::sqrt(6.0 / (kHid + kHid)),
                     b3 = std::sqrt(6.0 / (kHid + kOut));
        for (int i = 0; i < kWCount; ++i) {
            const double b = i < kW2 ? b1 : (i < kW3 ? b2 : b3);
            w[i] = (float)((uniform01(rs) * 2.0 - 1.0) * b);
        }
        st = copy_params(s, table.data(), w.data() + kW1, w.data() + kW2, w.data() + kW3, false);
        if (st == GI_OK) st = refresh_copies(s);
    }
    if (st != GI_OK) {
        nrc_free(s);
        delete s;
        return st;
    }
    *out = s;
    return GI_OK;
}

gi_status gi_nrc_destroy(gi_nrc_t nrc) {
    if (!nrc) return GI_OK;
    cudaDeviceSynchronize();
    nrc_free(nrc);
    delete nrc;
    return GI_OK;
}

gi_status gi_nrc_set_params(gi_nrc_t nrc, const float *table, const float *w1, const float *w2, const float *w3) {
    if (!nrc) {
        set_error("gi_nrc_set_params: NULL surrogate");
        return GI_ERR_INVALID_ARG;
    }
    gi_status st = cuda_status(cudaDeviceSynchronize(), "gi_nrc_set_params");
    if (st != GI_OK) return st;
    // reset Adam moments and gradients (the whole entry but the master features)
    st = table_field(nrc, nullptr, false, 2);
    if (st != GI_OK) return st;
    cudaError_t e = cudaMemset(nrc->grad, 0, (size_t)kL * nrc->T * sizeof(float2));
    if (e == cudaSuccess) e = cudaMemset(nrc->wm, 0, kWCount * 4);
    if (e == cudaSuccess) e = cudaMemset(nrc->wv, 0, kWCount * 4);
    if (e == cudaSuccess) e = cudaMemset(nrc->wg, 0, kWCount * 4);
    st = cuda_status(e, "gi_nrc_set_params");
    if (st == GI_OK) st = copy_params(nrc, table, w1, w2, w3, false);
    if (st == GI_OK) st = refresh_copies(nrc);
    nrc->steps = 0;
    return st;
}

gi_status gi_nrc_get_params(gi_nrc_t nrc, float *table, float *w1, float *w2, float *w3) {
    if (!nrc) {
        set_error("gi_nrc_get_params: NULL surrogate");
        return GI_ERR_INVALID_ARG;
    }
    return read_params(nrc, table, w1, w2, w3, false);
}

gi_status gi_nrc_set_gradients(gi_nrc_t nrc, const float *table, const float *w1, const float *w2, const float *w3) {
    if (!nrc) {
        set_error("gi_nrc_set_gradients: NULL surrogate");
        return GI_ERR_INVALID_ARG;
    }
    gi_status st = cuda_status(cudaDeviceSynchronize(), "gi_nrc_set_gradients");
    if (st == GI_OK) st = copy_params(nrc, table, w1, w2, w3, true);
    if (table) nrc->grads_set = true;
    return st;
}

gi_status gi_nrc_get_gradients(gi_nrc_t nrc, float *table, float *w1, float *w2, float *w3) {
    if (!nrc) {
        set_error("gi_nrc_get_gradients: NULL surrogate");
        return GI_ERR_INVALID_ARG;
    }
    return read_params(nrc, table, w1, w2, w3, true);
}

gi_status gi_nrc_infer(gi_nrc_t nrc, const gi_points *pts, float *out, gi_stream_t stream) {
    if (!nrc || !points_ok(pts) || (!out && pts->n)) {
        set_error("gi_nrc_infer: NULL argument or more than GI_NRC_MAX_BATCH points");
        return GI_ERR_INVALID_ARG;
    }
    if (pts->n == 0) return GI_OK;
    gi_status st = ensure_capacity(nrc, pts->n);
    if (st != GI_OK) return st;
    const cudaStream_t s = (cudaStream_t)stream;
    EncArgs e = enc_base(nrc);
    for (int a = 0; a < 3; ++a) {
        e.pos[a] = pts->pos[a];
        e.nrm[a] = pts->nrm[a];
    }
    e.n = pts->n;
    e.T = nullptr;
    // Plain launch: blocks scheduled while an earlier inference kernel (four CTAs of 47 KB per SM) is
    // resident would run with the little L1 that its shared memory leaves, and the table lookups live in
    // L1: repeated inferences took 55 us that way and take 42.4 this way.
    k_nrc_encode<kEncPoints><<<sample_blocks(nrc, pts->n), kEncThreads, 0, s>>>(e);
    st = cuda_status(cudaGetLastError(), "k_nrc_encode launch");
    if (st == GI_OK) st = launch_infer(nrc, pts->n, nullptr, reinterpret_cast<float4 *>(out), nullptr, s);
    return st;
}

gi_status gi_nrc_backward(gi_nrc_t nrc, const gi_points *pts, const float *const target[3], const float *mask,
                          uint32_t batch_norm, gi_stream_t stream) {
    if (!nrc || !points_ok(pts) || !target || (pts->n && (!target[0] || !target[1] || !target[2]))) {
        set_error("gi_nrc_backward: NULL argument or more than GI_NRC_MAX_BATCH points");
        return GI_ERR_INVALID_ARG;
    }
    const cudaStream_t s = (cudaStream_t)stream;
    gi_status st = cuda_status(cudaMemsetAsync(nrc->stats, 0, 16, s), "gi_nrc_backward");
    if (st != GI_OK || pts->n == 0) return st;
    st = ensure_capacity(nrc, pts->n);
    if (st != GI_OK) return st;
    EncArgs e = enc_base(nrc);
    for (int a = 0; a < 3; ++a) {
        e.pos[a] = pts->pos[a];
        e.nrm[a] = pts->nrm[a];
        e.target[a] = target[a];
    }
    e.mask = mask;
    e.n = pts->n;
    k_nrc_encode<kEncPoints><<<sample_blocks(nrc, pts->n), kEncThreads, 0, s>>>(e);
    st = cuda_status(cudaGetLastError(), "k_nrc_encode launch");
    const float B = (float)(batch_norm ? batch_norm : pts->n);
    nrc->last_minibatches = 1;
    int parts = 0;
    if (st == GI_OK) st = launch_train(nrc, pts->n, 2.0f / B, &parts, s);
    if (st == GI_OK) {
        launch(k_nrc_wgrad_reduce, (kWCount + 3 + 31) / 32, 256, 0, s, nrc->wpart, parts, nrc->wg, nrc->stats);
        st = cuda_status(cudaGetLastError(), "k_nrc_wgrad_reduce launch");
    }
    if (st == GI_OK) st = scatter_and_return(nrc, pts->pos, pts->nrm, nullptr, pts->n, s);
    return st;
}

gi_status gi_nrc_set_learning_rate(gi_nrc_t nrc, float lr) {
    if (!nrc || !(lr > 0.0f) || !std::isfinite(lr)) {
        set_error("gi_nrc_set_learning_rate: NULL surrogate or step size not finite and > 0");
        return GI_ERR_INVALID_ARG;
    }
    nrc->cfg.lr = lr;
    return GI_OK;
}

// One Adam step; parts: rows of s->wpart whose sums belong to the step's weight gradients and losses.
static gi_status adam_step(gi_nrc_s *nrc, int parts, cudaStream_t s) {
    nrc->steps += 1;
    const double t = (double)nrc->steps;
    AdamArgs a;
    a.lr = nrc->cfg.lr;
    a.b1 = nrc->cfg.beta1;
    a.b2 = nrc->cfg.beta2;
    a.eps = nrc->cfg.adam_eps;
    a.c1 = (float)(1.0 - std::pow((double)nrc->cfg.beta1, t));
    a.c2 = (float)(1.0 - std::pow((double)nrc->cfg.beta2, t));
    AdamTableArgs at;
    at.tab = nrc->tab;
    at.grad = nrc->grad;
    at.tab16 = nrc->tab16;
    at.log2_table = nrc->cfg.log2_table;
    const uint32_t resident = (uint32_t)nrc->sms * kAdamBlocksPerSm * kAdamWarps;
    const uint32_t chunk = ((uint64_t)kL << nrc->cfg.log2_table) <= 128ull * resident ? 64u : 256u;
    at.chunk0[0] = 0;
    for (int l = 0; l < kL; ++l) {
        // a dense level's samples reach its first 6 (R + 1)^3 entries; gradients the caller wrote, all
        const uint64_t V = (uint64_t)nrc->geo.lv.res[l] + 1u;
        const uint64_t used = nrc->geo.lv.dense[l] && !nrc->grads_set ? 6u * V * V * V : nrc->T;
        at.chunk0[l + 1] = at.chunk0[l] + (uint32_t)((used + chunk - 1) / chunk);
    }
    nrc->grads_set = false;
    const AdamWeightArgs aw = {nrc->w, nrc->wm, nrc->wv, nrc->wg, nrc->wimg, nrc->wpart, parts, nrc->stats};
    const unsigned blocks = std::min<uint32_t>((at.chunk0[kL] + kAdamWarps - 1) / kAdamWarps, (uint32_t)nrc->sms * kAdamBlocksPerSm);
    launch(chunk == 64u ? k_nrc_adam<64> : k_nrc_adam<256>, kAdamWBlocks + blocks, 32 * kAdamWarps, 0, s, at, aw, a);
    return cuda_status(cudaGetLastError(), "k_nrc_adam launch");
}

gi_status gi_nrc_adam(gi_nrc_t nrc, gi_stream_t stream) {
    if (!nrc) {
        set_error("gi_nrc_adam: NULL surrogate");
        return GI_ERR_INVALID_ARG;
    }
    return adam_step(nrc, 0, (cudaStream_t)stream);
}

gi_status gi_nrc_train_frame(gi_nrc_t nrc, gi_cache_t cache, const gi_hits *hits, const uint32_t *slot_ids,
                             uint32_t frame, gi_stream_t stream) {
    if (!nrc || !cache || !hits || !slot_ids || !hits->ray_len || hits->n == 0 || hits->n > nrc->cfg.max_records ||
        hits->n > 0xFFFFFFFFull) {
        set_error("gi_nrc_train_frame: NULL argument, no records, or more than max_records");
        return GI_ERR_INVALID_ARG;
    }
    for (int a = 0; a < 3; ++a)
        if (!hits->pos[a] || !hits->nrm[a]) {
            set_error("gi_nrc_train_frame: NULL record plane");
            return GI_ERR_INVALID_ARG;
        }
    const cudaStream_t s = (cudaStream_t)stream;
    gi_status st = cuda_status(cudaMemsetAsync(nrc->stats, 0, 16, s), "gi_nrc_train_frame");
    if (st != GI_OK) return st;
    const uint32_t steps = nrc->cfg.train_steps, B = nrc->cfg.batch / steps;
    EncArgs e = enc_base(nrc);
    for (int a = 0; a < 3; ++a) {
        e.pos[a] = hits->pos[a];
        e.nrm[a] = hits->nrm[a];
    }
    e.len = hits->ray_len;
    e.n = B;
    e.n_records = (uint32_t)hits->n;
    e.seed = pcg_hash(frame + 1u);
    e.slot_ids = slot_ids;
    e.cv = cache_view(cache);
    for (uint32_t j = 0; j < steps && st == GI_OK; ++j) {
        e.offset = j * B;
        launch(k_nrc_encode<kEncSampled>, sample_blocks(nrc, B), kEncThreads, 0, s, e);
        st = cuda_status(cudaGetLastError(), "k_nrc_encode launch");
        int parts = 0;
        if (st == GI_OK) st = launch_train(nrc, B, 2.0f / (float)B, &parts, s);
        if (st == GI_OK) st = scatter_and_return(nrc, hits->pos, hits->nrm, nrc->idx, B, s);
        if (st == GI_OK) st = adam_step(nrc, parts, s);
    }
    nrc->last_minibatches = steps;
    return st;
}

gi_status gi_nrc_query_frame(gi_nrc_t nrc, gi_cache_t cache, const gi_hits *hits, const uint32_t *slot_ids,
                             const gi_view *view, gi_stream_t stream) {
    if (!nrc || !cache || !hits || !slot_ids || !hits->ray_len || !view_ok(view) || hits->n > nrc->cfg.max_records) {
        set_error("gi_nrc_query_frame: NULL argument, bad view, or more than max_records");
        return GI_ERR_INVALID_ARG;
    }
    for (int a = 0; a < 3; ++a)
        if (!hits->pos[a] || !hits->nrm[a]) {
            set_error("gi_nrc_query_frame: NULL record plane");
            return GI_ERR_INVALID_ARG;
        }
    const cudaStream_t s = (cudaStream_t)stream;
    gi_status st = cuda_status(cudaMemsetAsync(nrc->qcount, 0, 4, s), "gi_nrc_query_frame");
    if (st != GI_OK) return st;
    nrc->queried = true;
    nrc->last_query_n = hits->n;
    if (hits->n == 0) return GI_OK;
    SelectArgs a;
    for (int k = 0; k < 3; ++k) a.pos[k] = hits->pos[k];
    a.len = hits->ray_len;
    a.slot_ids = slot_ids;
    a.n = (uint32_t)hits->n;
    a.cv = cache_view(cache);
    a.kp = cache_update_args(cache, hits, view, nullptr).kp;
    a.query_lod = nrc->cfg.query_lod;
    a.trust = nrc->cfg.trust;
    a.trained = nrc->steps > 0 ? 1u : 0u;
    a.stats = nrc->stats;
    a.max_q = nrc->cfg.max_queries;
    a.qidx = nrc->qidx;
    a.qcount = nrc->qcount;
    a.bits = nrc->bits;
    const uint32_t words = (a.n + 31u) / 32u;
    const uint32_t per = kSelWarps * kSelWords;
    const unsigned blocks = std::min<uint32_t>((words + per - 1) / per, (uint32_t)nrc->sms * 8);
    launch(k_nrc_select, blocks, 32 * kSelWarps, 0, s, a);
    st = cuda_status(cudaGetLastError(), "k_nrc_select launch");
    if (st != GI_OK || nrc->cfg.max_queries == 0) return st;
    EncArgs e = enc_base(nrc);
    for (int k = 0; k < 3; ++k) {
        e.pos[k] = hits->pos[k];
        e.nrm[k] = hits->nrm[k];
    }
    e.len = hits->ray_len;
    e.n = nrc->cfg.max_queries;
    e.qidx = nrc->qidx;
    e.qcount = nrc->qcount;
    e.T = nullptr;
    launch(k_nrc_encode_queries, (unsigned)(nrc->sms * kEncBlocksPerSm), kEncThreads, 0, s, e);
    st = cuda_status(cudaGetLastError(), "k_nrc_encode launch");
    if (st == GI_OK) st = launch_infer(nrc, nrc->cfg.max_queries, nrc->qcount, nrc->ovr, nrc->qidx, s);
    return st;
}

gi_status gi_nrc_answers(gi_nrc_t nrc, uint32_t *records, float *rad, uint32_t capacity, uint32_t *count,
                         gi_stream_t stream) {
    if (!nrc || !count || (capacity && (!records || !rad))) {
        set_error("gi_nrc_answers: NULL argument");
        return GI_ERR_INVALID_ARG;
    }
    const cudaStream_t s = (cudaStream_t)stream;
    uint32_t c = 0;
    gi_status st = cuda_status(cudaStreamSynchronize(s), "gi_nrc_answers");
    if (st == GI_OK) st = cuda_status(cudaMemcpy(&c, nrc->qcount, 4, cudaMemcpyDeviceToHost), "gi_nrc_answers");
    if (st != GI_OK) return st;
    c = std::min(c, nrc->cfg.max_queries);
    *count = c;
    if (capacity == 0 && !records) return GI_OK;
    if (c > capacity) {
        set_error("gi_nrc_answers: %u answers, capacity %u", c, capacity);
        return GI_ERR_CAPACITY;
    }
    if (c) {
        k_nrc_gather_answers<<<(c + 255) / 256, 256, 0, s>>>(nrc->qidx, nrc->ovr, c, records,
                                                               reinterpret_cast<float4 *>(rad));
        st = cuda_status(cudaGetLastError(), "k_nrc_gather_answers launch");
        if (st == GI_OK) st = cuda_status(cudaStreamSynchronize(s), "gi_nrc_answers");
    }
    return st;
}

gi_status gi_nrc_stats(gi_nrc_t nrc, gi_nrc_stats_t *out, gi_stream_t stream) {
    if (!nrc || !out) {
        set_error("gi_nrc_stats: NULL argument");
        return GI_ERR_INVALID_ARG;
    }
    float st4[4];
    uint32_t q = 0, err = 0;
    gi_status st = cuda_status(cudaStreamSynchronize((cudaStream_t)stream), "gi_nrc_stats");
    if (st == GI_OK) st = cuda_status(cudaMemcpy(st4, nrc->stats, 16, cudaMemcpyDeviceToHost), "gi_nrc_stats");
    if (st == GI_OK) st = cuda_status(cudaMemcpy(&q, nrc->qcount, 4, cudaMemcpyDeviceToHost), "gi_nrc_stats");
    if (st == GI_OK) st = cuda_status(cudaMemcpy(&err, nrc->err, 4, cudaMemcpyDeviceToHost), "gi_nrc_stats");
    if (st != GI_OK) return st;
    out->steps = nrc->steps;
    out->loss = st4[0] / (float)nrc->last_minibatches;
    out->judged_error = st4[2] > 0.f ? st4[1] / st4[2] : 0.f;
    out->trusted = (nrc->steps > 0 && st4[2] > 0.f && st4[1] <= nrc->cfg.trust * st4[2]) ? 1u : 0u;
    out->queries = nrc->queried ? std::min(q, nrc->cfg.max_queries) : 0u;
    if (err) {
        set_error("gi_nrc: a bounded tensor-core wait ran out (error word %u)", err);
        return GI_ERR_TIMEOUT;
    }
    return GI_OK;
}

}  // extern "C"
