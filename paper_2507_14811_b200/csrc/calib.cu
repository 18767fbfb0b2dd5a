// Min/max calibration (Sec. 4.3.2 scale formula; strict min/max, App. B sensitivity analysis):
// per K-segment extrema of a calibration batch, or per (K-segment, N-segment) abs-max of a weight
// matrix, reduced through ordered-integer atomics into workspace partials, then one IEEE division
// per scale, in one launch.
#include <cuda_bf16.h>
#include <mutex>
#include "sq_common.cuh"

namespace sq {
namespace {

constexpr int kWarps = 8;
constexpr int kThreads = kWarps * 32;
constexpr int kRowsInFlight = 8;         // rows whose loads a warp issues before it uses the first

// monotone map float -> uint32 (a < b  <=>  enc(a) < enc(b)); 0 is never produced by inputs other than NaNs.  A
// minimum is kept as the maximum of ~enc, which no input maps to 0 either, so one neutral value, 0, serves both
// slots of a partial.
__device__ __forceinline__ uint32_t enc(float f)
{
    uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float dec(uint32_t u)
{
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7FFFFFFFu) : ~u);
}

__device__ __forceinline__ float ld1(const float *p) { return __ldg(p); }
__device__ __forceinline__ float ld1(const __nv_bfloat16 *p)
{
    return __uint_as_float(uint32_t(__ldg(reinterpret_cast<const unsigned short *>(p))) << 16);
}

// Running extrema of the columns of one 16-byte piece of a row: 4 fp32 columns, or 8 bf16 columns as 4 packed pairs
// (two per instruction).  Every column keeps its own extrema, so a piece that straddles a K-segment bound needs
// nothing special until the end.  NaNs lose against any number, as with fmaxf / fminf.
template <typename Tin> struct Extrema;
template <> struct Extrema<float> {
    static constexpr int kCols = 4;
    float mx[4], mn[4];
    __device__ __forceinline__ void reset()
    {
#pragma unroll
        for (int i = 0; i < 4; i++) { mx[i] = -INFINITY; mn[i] = INFINITY; }
    }
    __device__ __forceinline__ void add(uint4 w)
    {
        const float v[4] = {__uint_as_float(w.x), __uint_as_float(w.y), __uint_as_float(w.z), __uint_as_float(w.w)};
#pragma unroll
        for (int i = 0; i < 4; i++) { mx[i] = fmaxf(mx[i], v[i]); mn[i] = fminf(mn[i], v[i]); }
    }
    __device__ __forceinline__ void add1(int col, float v) { mx[col] = fmaxf(mx[col], v); mn[col] = fminf(mn[col], v); }
    __device__ __forceinline__ float hi(int col) const { return mx[col]; }
    __device__ __forceinline__ float lo(int col) const { return mn[col]; }
};
template <> struct Extrema<__nv_bfloat16> {
    static constexpr int kCols = 8;
    __nv_bfloat162 mx[4], mn[4];
    __device__ __forceinline__ void reset()
    {
#pragma unroll
        for (int i = 0; i < 4; i++) {
            mx[i] = __float2bfloat162_rn(-INFINITY);
            mn[i] = __float2bfloat162_rn(INFINITY);
        }
    }
    __device__ __forceinline__ void add(uint4 w)
    {
        const uint32_t v[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const __nv_bfloat162 x = *reinterpret_cast<const __nv_bfloat162 *>(&v[i]);
            mx[i] = __hmax2(mx[i], x);
            mn[i] = __hmin2(mn[i], x);
        }
    }
    __device__ __forceinline__ void add1(int col, float v)                 // v is a bf16 value: exact
    {
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const __nv_bfloat16 x = __float2bfloat16_rn(v);
            if (col == 2 * i) { mx[i].x = __hmax(mx[i].x, x); mn[i].x = __hmin(mn[i].x, x); }
            if (col == 2 * i + 1) { mx[i].y = __hmax(mx[i].y, x); mn[i].y = __hmin(mn[i].y, x); }
        }
    }
    __device__ __forceinline__ float hi(int col) const { return __bfloat162float(col & 1 ? mx[col >> 1].y : mx[col >> 1].x); }
    __device__ __forceinline__ float lo(int col) const { return __bfloat162float(col & 1 ? mn[col >> 1].y : mn[col >> 1].x); }
};

enum : int { kScaleSingle = 0, kScaleDual = 1, kScaleZeroPoint = 2 };

struct CalibOut {
    int kind;
    float q_max, q_min_abs;
    float *s_pos, *s_neg;        // zero-point mode: s_pos is s_x
    int32_t *z_x;
};

// Scales of one (K-segment, N-segment) block from its extrema (0 in either slot: nothing seen).
// Zero-point mode (App. A asymmetric quantizer): s = (hi - lo) / 255 and z = -128 - round(lo / s) from the extrema
// widened to contain 0 (one fp32 subtraction, two IEEE divisions, round half to even); a zero range gives s = 1, z = 0.
__device__ __forceinline__ void finalize_block(int i, uint32_t emx, uint32_t emn_inv, const CalibOut &out)
{
    const float mx = (emx == 0u || emx == enc(-INFINITY)) ? 0.0f : dec(emx);
    const float mn = (emn_inv == 0u || ~emn_inv == enc(INFINITY)) ? 0.0f : dec(~emn_inv);
    if (out.kind == kScaleZeroPoint) {
        const float hi = fmaxf(mx, 0.0f), lo = fminf(mn, 0.0f);
        const float range = __fsub_rn(hi, lo);
        if (range > 0.0f) {
            const float s = __fdiv_rn(range, 255.0f);
            const float zf = __fsub_rn(-128.0f, rintf(__fdiv_rn(lo, s)));
            out.s_pos[i] = s;
            out.z_x[i] = int(fminf(fmaxf(zf, -128.0f), 127.0f));
        } else {
            out.s_pos[i] = 1.0f;
            out.z_x[i] = 0;
        }
    } else if (out.kind == kScaleDual) {
        const float hi = fmaxf(mx, 0.0f), lo = fmaxf(-mn, 0.0f);
        out.s_pos[i] = hi > 0.0f ? __fdiv_rn(hi, out.q_max) : 1.0f;
        out.s_neg[i] = lo > 0.0f ? __fdiv_rn(lo, out.q_min_abs) : 1.0f;
    } else {
        const float a = fmaxf(fabsf(mx), fabsf(mn));
        out.s_pos[i] = a > 0.0f ? __fdiv_rn(a, out.q_max) : 1.0f;
    }
}

// Extrema and scales in one launch.  HBM-bound on weight matrices, latency-bound on calibration batches.  A block
// takes 32 16-byte pieces of a row (512 consecutive bytes per warp and row) and a contiguous range of rows, its
// eight warps every eighth of them with kRowsInFlight rows' loads outstanding; the host cuts the rows so that the
// grid is one full wave, or, for small inputs, so that a warp's rows are all in flight at once.  Extrema stay in
// registers until the rows leave their N-segment, then go through a warp shuffle (where the warp's columns lie in one
// K-segment) into shared and from there into global words per block, and the last block of the grid to finish
// makes the scales.  Nothing waits.  The words and the arrival count are cleared by a fill in front of the kernel.
// (18432 x 3072 fp32 weights: 147 us with one column per thread, element-wide loads and separate set-up and
// scale launches, 40 us now = 5.6 TB/s; a 256 x 3072 bf16 batch 18.9 -> 8.2 us, fill included.)
template <typename Tin>
__global__ void __launch_bounds__(kThreads, 5)
calib_kernel(const Tin *__restrict__ X, int64_t rows, int K, int64_t ld, const __grid_constant__ SegBounds sb, int is_weight,
             int64_t rows_per_block, uint32_t *__restrict__ partials, uint32_t *__restrict__ done_count, CalibOut out)
{
    constexpr int kCols = Extrema<Tin>::kCols;
    __shared__ uint32_t sh[2 * kMaxBlocks];                   // {max, inverted min} per block
    __shared__ uint32_t sh_last;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int Qs = is_weight ? sb.Q : 1;
    const int nblk = sb.P * Qs;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < 2 * nblk; i += kThreads) sh[i] = 0u;
    __syncthreads();

    const int k0 = (int(blockIdx.x) * 32 + lane) * kCols;
    const int ncols = min(kCols, K - k0);                     // <= 0: this lane has no columns
    const int64_t r0 = int64_t(blockIdx.y) * rows_per_block;
    const int64_t r1 = min(rows, r0 + rows_per_block);
    int p0 = 0;                                               // K-segment of the first column
    while (p0 + 1 < sb.P && k0 >= sb.kb[p0 + 1]) p0++;
    const bool whole = ncols == kCols && k0 + kCols <= sb.kb[p0 + 1];
    const int p_first = __shfl_sync(0xFFFFFFFFu, p0, 0);
    const bool uniform = __all_sync(0xFFFFFFFFu, ncols <= 0 || (whole && p0 == p_first));
    int q = 0;
    if (is_weight) while (q + 1 < sb.Q && r0 >= sb.nb[q + 1]) q++;

    for (int64_t ra = r0; ra < r1;) {
        const int64_t rb = is_weight ? min(r1, int64_t(sb.nb[q + 1])) : r1;      // rows of one N-segment
        Extrema<Tin> e;
        e.reset();
        const Tin *src = X + k0;
        if (ncols == kCols) {
            int64_t r = ra + warp;
            for (; r + int64_t(kRowsInFlight - 1) * kWarps < rb; r += int64_t(kRowsInFlight) * kWarps) {
                uint4 v[kRowsInFlight];
#pragma unroll
                for (int u = 0; u < kRowsInFlight; u++)
                    v[u] = __ldg(reinterpret_cast<const uint4 *>(src + (r + int64_t(u) * kWarps) * ld));
#pragma unroll
                for (int u = 0; u < kRowsInFlight; u++) e.add(v[u]);
            }
            if (r < rb) {                                     // fewer rows left: the last one again instead of a branch per load
                uint4 v[kRowsInFlight];
#pragma unroll
                for (int u = 0; u < kRowsInFlight; u++)
                    v[u] = __ldg(reinterpret_cast<const uint4 *>(src + min(r + int64_t(u) * kWarps, rb - 1) * ld));
#pragma unroll
                for (int u = 0; u < kRowsInFlight; u++) e.add(v[u]);
            }
        } else if (ncols > 0) {                               // the row's last columns: nothing beyond K is read
            for (int64_t r = ra + warp; r < rb; r += kWarps)
                for (int c = 0; c < ncols; c++) e.add1(c, ld1(src + r * ld + c));
        }
        if (uniform) {
            float mx = e.hi(0), mn = e.lo(0);
#pragma unroll
            for (int c = 1; c < kCols; c++) { mx = fmaxf(mx, e.hi(c)); mn = fminf(mn, e.lo(c)); }
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) {
                mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
                mn = fminf(mn, __shfl_xor_sync(0xFFFFFFFFu, mn, o));
            }
            if (lane == 0) {
                atomicMax(&sh[2 * (p_first * Qs + q)], enc(mx));
                atomicMax(&sh[2 * (p_first * Qs + q) + 1], ~enc(mn));
            }
        } else if (ncols > 0) {
            // a lane's columns of one K-segment go out together: neighbouring lanes update the same words, one after the other
            // (4096 x 3072 bf16 weights in 64 x 64 segments, call included: 41.9 us with an update per column, 27.3 now)
            int p = p0;
            float mx = e.hi(0), mn = e.lo(0);
            auto put = [&] {
                atomicMax(&sh[2 * (p * Qs + q)], enc(mx));
                atomicMax(&sh[2 * (p * Qs + q) + 1], ~enc(mn));
            };
#pragma unroll
            for (int c = 1; c < kCols; c++) {
                if (c < ncols) {
                    if (p + 1 < sb.P && k0 + c >= sb.kb[p + 1]) {          // bounds ascend: the next column is in the next segment
                        put();
                        p++;
                        mx = e.hi(c);
                        mn = e.lo(c);
                    } else {
                        mx = fmaxf(mx, e.hi(c));
                        mn = fminf(mn, e.lo(c));
                    }
                }
            }
            put();
        }
        ra = rb;
        if (is_weight && ra < r1) q++;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 2 * nblk; i += kThreads)
        if (sh[i] != 0u) atomicMax(&partials[i], sh[i]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) sh_last = atomicAdd(done_count, 1u) == gridDim.x * gridDim.y - 1u ? 1u : 0u;
    __syncthreads();
    if (sh_last) {                                            // every other block's extrema are in `partials`
        __threadfence();
        for (int i = threadIdx.x; i < nblk; i += kThreads)
            finalize_block(i, __ldcg(&partials[2 * i]), __ldcg(&partials[2 * i + 1]), out);
    }
}

// Launch shape; false if the matrix is beyond what one grid covers (checked before any launch).  The bound on K is the
// one the entry points document; a grid of 2^31 - 1 blocks covers everything below it.
template <typename Tin>
bool calib_grid(int64_t rows, int64_t K, int sms, dim3 *grid, int64_t *rows_per_block)
{
    if (rows < 1 || K < 1 || rows > (int64_t(0x7FFFFFFF) << 6) || K > int64_t(65535) * 256) return false;
    constexpr int64_t cols = 32 * Extrema<Tin>::kCols;
    const int64_t gx = (K + cols - 1) / cols;
    // one wave of five blocks per SM; at least kRowsInFlight rows per warp
    int64_t gy = (int64_t(sms) * 5) / gx;
    const int64_t most = (rows + kWarps * kRowsInFlight - 1) / (kWarps * kRowsInFlight);
    if (gy > most) gy = most;
    if (gy < 1) gy = 1;
    if (gy > 65535) gy = 65535;
    const int64_t per = (rows + gy - 1) / gy;
    *rows_per_block = per;
    *grid = dim3(unsigned(gx), unsigned((rows + per - 1) / per));
    return true;
}

template <typename Tin>
sq_status launch_calib_t(const Tin *X, int64_t rows, int64_t K, int64_t ld, const SegBounds &sb, int is_weight,
                         uint32_t *partials, uint32_t *done_count, const CalibOut &out, cudaStream_t st)
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
        return SQ_ERR_CUDA;
    dim3 grid;
    int64_t rows_per_block = 0;
    if (!calib_grid<Tin>(rows, K, sms, &grid, &rows_per_block)) return SQ_ERR_SHAPE;      // nothing has been launched yet
    // the arrival count and the partials lie in one piece of memory: one fill readies both, whatever is in them
    const int nblk = sb.P * (is_weight ? sb.Q : 1);
    uint8_t *state = reinterpret_cast<uint8_t *>(done_count);
    cudaError_t e = cudaMemsetAsync(state, 0, size_t(reinterpret_cast<uint8_t *>(partials + 2 * nblk) - state), st);
    if (e != cudaSuccess) { note_cuda_error(e); return SQ_ERR_CUDA; }
    calib_kernel<Tin><<<grid, kThreads, 0, st>>>(X, rows, int(K), ld, sb, is_weight, rows_per_block, partials, done_count, out);
    count_launch();
    e = cudaGetLastError();
    if (e != cudaSuccess) { note_cuda_error(e); return SQ_ERR_CUDA; }
    return SQ_OK;
}

sq_status launch_calib_any(const void *X, sq_dtype dt, int64_t rows, int64_t K, int64_t ld, const SegBounds &sb,
                           int is_weight, uint32_t *partials, uint32_t *done_count, const CalibOut &out, cudaStream_t st)
{
    return dt == SQ_F32 ? launch_calib_t(static_cast<const float *>(X), rows, K, ld, sb, is_weight, partials, done_count, out, st)
                        : launch_calib_t(static_cast<const __nv_bfloat16 *>(X), rows, K, ld, sb, is_weight, partials, done_count, out, st);
}

}  // namespace

sq_status launch_calib(const void *X, sq_dtype dt, int64_t rows, int64_t K, int64_t ld, const SegBounds &sb,
                       int is_weight, int dual, float q_max, float q_min_abs, float *s_pos, float *s_neg,
                       uint32_t *partials, uint32_t *done_count, cudaStream_t st)
{
    const CalibOut out{!is_weight && dual ? kScaleDual : kScaleSingle, q_max, q_min_abs, s_pos, s_neg, nullptr};
    return launch_calib_any(X, dt, rows, K, ld, sb, is_weight, partials, done_count, out, st);
}

sq_status launch_calib_zero_point(const void *X, sq_dtype dt, int64_t rows, int64_t K, int64_t ld, const SegBounds &sb,
                                  float *s_x, int32_t *z_x, uint32_t *partials, uint32_t *done_count, cudaStream_t st)
{
    const CalibOut out{kScaleZeroPoint, 0.0f, 0.0f, s_x, nullptr, z_x};
    return launch_calib_any(X, dt, rows, K, ld, sb, 0, partials, done_count, out, st);
}

namespace {

// ----------------------------------------------------------------------------- built-in scratch
// Reduction partials for callers that have no device allocator to take a workspace from: 2 words per
// (K-segment, N-segment) block, SQ_STATIC_CALIB_MAX_BLOCKS blocks, 8 KiB, behind the arrival count.  The array lives in the
// library's device image, so every GPU that loads the library holds it until the process exits, and
// every call on that GPU shares it.
static __device__ __align__(256) uint32_t g_static_partials[2 + SQ_STATIC_CALIB_MAX_BLOCKS * 2];   // arrival count first

// In host code the name g_static_partials is only a handle for the runtime; the device address has
// to be asked for, once per device, with that device current.
static sq_status static_partials_address(uint32_t **out)
{
    constexpr int kMaxDevices = 64;
    static std::mutex mu;
    static uint32_t *addr[kMaxDevices] = {};
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return SQ_ERR_CUDA;
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_static_partials) != cudaSuccess || !p) return SQ_ERR_CUDA;
        addr[dev] = static_cast<uint32_t *>(p);
    }
    *out = addr[dev];
    return SQ_OK;
}

}  // namespace

sq_status launch_calib_static(const void *X, sq_dtype dt, int64_t rows, int64_t K, int64_t ld, const SegBounds &sb,
                              int is_weight, int dual, float q_max, float q_min_abs, float *s_pos, float *s_neg,
                              cudaStream_t st)
{
    if (sb.P * (is_weight ? sb.Q : 1) > SQ_STATIC_CALIB_MAX_BLOCKS) return SQ_ERR_UNSUPPORTED;
    uint32_t *partials = nullptr;
    const sq_status r = static_partials_address(&partials);
    if (r != SQ_OK) return r;
    // launch_calib clears the partials it is going to use, so the previous call's contents never leak into this one
    return launch_calib(X, dt, rows, K, ld, sb, is_weight, dual, q_max, q_min_abs, s_pos, s_neg, partials + 2, partials, st);
}

}  // namespace sq
