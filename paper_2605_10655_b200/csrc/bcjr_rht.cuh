// Incoherence processing around the trellis pass (Section 3.1; Section 4, "Quantization
// configuration"): a random-sign Hadamard rotation on both sides of the weight matrix and a scale
// per group of 16 elements.  The paper names both without formulas; the forms used are
//     W~ = H_m diag(sL) W diag(sR) H_n / sqrt(m n),      W = diag(sL) H_m W~ H_n diag(sR) / sqrt(m n)
// with Sylvester-ordered Walsh-Hadamard matrices (entries +-1, H H = size I), and
//     scale(group) = sqrt(mean of the 16 squares),  W_scaled = W / scale.
// All of it is one or a few passes over the matrix: bound by HBM / L2 bandwidth.
//
// Fast Walsh-Hadamard transform.  The rotation of a row-major matrix is ONE transform over the bits of the linear index, and
// any subset of the bits can be taken in any order.  A matrix of 2^14 elements or more takes two kernels: the low 14 bits
// (the row transform and the lowest column bits: contiguous tiles of 64 KB, fwht_tile_kernel), then the remaining row-index bits,
// ten at a time (tiles of 2^B rows x 16 columns or more: fwht_next_kernel, beyond 2^24 elements then fwht_cols_kernel).  Each reads and writes the matrix once.  A thread
// holds 32 elements and runs five butterfly stages on them in registers, so that a tile passes through shared memory twice
// in the first kernel and once in the second.  Smaller matrices are one radix-8 transform in shared memory
// (fwht_small_kernel).  8192 x 2048, rotation and its inverse with group scales between: 313 -> 170 us
// (a pass over the matrix for every three bits before), 160 with addresses that are constants, 146 with streaming loads (rht_stream4).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace bcjr {

// Four floats that this kernel is the last to want for a while: their lines go first when the L2 needs room, so that what the kernel
// writes is still there for the next one (a 67 MB matrix and its image do not both fit 126 MB).
__device__ __forceinline__ uint64_t rht_stream_policy()
{
    uint64_t policy;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    return policy;
}
__device__ __forceinline__ float4 rht_stream4(const float4 *p, uint64_t policy)
{
    float4 v;
    asm volatile("ld.global.L1::no_allocate.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p), "l"(policy) : "memory");
    return v;
}

// stages for bits s with first <= s < 3 of an 8-point transform (first = 0: all three)
template <typename T>
__device__ __forceinline__ void fwht8(T (&v)[8], int first)
{
    if (first <= 0) {
#pragma unroll
        for (int j = 0; j < 8; j += 2) { const T a = v[j], b = v[j + 1]; v[j] = a + b; v[j + 1] = a - b; }
    }
    if (first <= 1) {
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (!(j & 2)) { const T a = v[j], b = v[j + 2]; v[j] = a + b; v[j + 2] = a - b; }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) { const T a = v[j], b = v[j + 4]; v[j] = a + b; v[j + 4] = a - b; }
}

// shared-memory index with eight floats of padding per 64: keeps the stride-8 pass off a single bank group
__device__ __forceinline__ int rht_pad(int i) { return i + ((i >> 6) << 3); }

// Signs of element `at` of a matrix of 2^ln columns.
struct RhtSigns {
    const float *rows, *cols;
    int ln;
    __device__ __forceinline__ float of(int64_t at) const { return __ldg(cols + (at & (((int64_t)1 << ln) - 1))) * __ldg(rows + (at >> ln)); }
};

// The whole matrix of 2^LOGN <= 2^13 elements: out = WHT(in * (pre ? signs : 1)) * scale * (pre ? 1 : signs), one block of 2^LOGN / 8 threads
template <int LOGN>
__global__ void fwht_small_kernel(const float *in, float *out, RhtSigns s, float scale, int pre)
{
    constexpr int N = 1 << LOGN;
    extern __shared__ float row[];
    const int t = threadIdx.x;
    float v[8];
    // plain loads: `out` may be `in` (in place), so the matrix is not read-only for the kernel
    const float4 a = reinterpret_cast<const float4 *>(in)[2 * t], b = reinterpret_cast<const float4 *>(in)[2 * t + 1];
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    if (pre) {
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] *= s.of(8 * t + j);
    }
    fwht8(v, 0);
    float *p = row + rht_pad(8 * t);
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    *reinterpret_cast<float4 *>(p + 4) = make_float4(v[4], v[5], v[6], v[7]);
    __syncthreads();
    // full radix-8 passes on bits [o, o+3), then one last pass on the top three bits that runs only the stages not done yet
    for (int o = 3;; o += 3) {
        const bool last = o + 3 >= LOGN;
        const int oo = last ? LOGN - 3 : o;                     // bit offset of this pass
        const int first = o - oo;                                // stages below `first` were done by earlier passes
        const int lo = t & ((1 << oo) - 1), hi = t >> oo;
        const int base = (hi << (oo + 3)) | lo;
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = row[rht_pad(base + (j << oo))];
        fwht8(v, first);
        if (last) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int i = base + (j << oo);
                out[i] = v[j] * scale * (pre ? 1.f : s.of(i));
            }
            break;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) row[rht_pad(base + (j << oo))] = v[j];
        __syncthreads();
    }
}

// butterfly stages on every index bit of v[2^N], strides 1 .. 2^(N-1)
template <int N>
__device__ __forceinline__ void fwht_reg(float (&v)[1 << N])
{
#pragma unroll
    for (int h = 1; h < (1 << N); h <<= 1)
#pragma unroll
        for (int j = 0; j < (1 << N); ++j)
            if (!(j & h)) { const float a = v[j], b = v[j + h]; v[j] = a + b; v[j + h] = a - b; }
}

constexpr int RHT_TILE_BITS = 14, RHT_THREADS = 512;
constexpr size_t RHT_TILE_SMEM = ((size_t)(1 << RHT_TILE_BITS) + (1 << (RHT_TILE_BITS - 5))) * 4;
// four floats of padding per 128: the lanes of the second pass differ in bits 0, 1 and 7 .. 9
__device__ __forceinline__ int rht_tile_pad(int e) { return e + ((e >> 7) << 2); }

// Index bits 0 .. 13 of tile blockIdx.x (2^14 consecutive elements).  MODE 1: inputs times their signs; 2: outputs.
template <int MODE>
__global__ void __launch_bounds__(RHT_THREADS, 2) fwht_tile_kernel(const float *in, float *out, RhtSigns s, float scale)
{
    extern __shared__ __align__(16) float tile[];
    const int t = threadIdx.x;
    const int64_t base = (int64_t)blockIdx.x << RHT_TILE_BITS;
    const uint64_t policy = rht_stream_policy();
    float v[32];
    // bits 0, 1 (inside a float4) and 11 .. 13: element 4 (t + 512 i) + j
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float4 f = rht_stream4(reinterpret_cast<const float4 *>(in + base) + t + 512 * i, policy);
        v[4 * i] = f.x; v[4 * i + 1] = f.y; v[4 * i + 2] = f.z; v[4 * i + 3] = f.w;
    }
    if (MODE == 1) {
        const int cm = (1 << s.ln) - 1;
        const float *rows = s.rows + (base >> s.ln);             // (a tile starts with a row, or inside one: then it has no other)
        const int in_row = (int)(base & cm);
        float4 c = __ldg(reinterpret_cast<const float4 *>(s.cols + ((in_row + 4 * t) & cm)));
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (i > 0 && s.ln > 11) c = __ldg(reinterpret_cast<const float4 *>(s.cols + ((in_row + 4 * t + 2048 * i) & cm)));
            const float r = __ldg(rows + ((in_row + 4 * t + 2048 * i) >> s.ln));
            v[4 * i] *= c.x * r; v[4 * i + 1] *= c.y * r; v[4 * i + 2] *= c.z * r; v[4 * i + 3] *= c.w * r;
        }
    }
    fwht_reg<5>(v);
    float *p1 = tile + rht_tile_pad(4 * t);                      // (the padding is linear in the bits of i and j below)
#pragma unroll
    for (int i = 0; i < 8; ++i) *reinterpret_cast<float4 *>(p1 + i * (2048 + 64)) = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    __syncthreads();
    // bits 2 .. 6
    {
        float *p = tile + rht_tile_pad((t & 3) | ((t >> 2) << 7));
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = p[j << 2];
        fwht_reg<5>(v);
#pragma unroll
        for (int j = 0; j < 32; ++j) p[j << 2] = v[j];
    }
    __syncthreads();
    // bits 7 .. 10, for both values of bit 13
    const int e0 = (t & 127) | (((t >> 7) & 3) << 11);
    const float *p3 = tile + rht_tile_pad(e0);
    float *q = out + base + e0;
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        float u[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) u[j] = p3[j * (128 + 4) + x * (8192 + 256)];
        fwht_reg<4>(u);
        if (MODE == 2) {
#pragma unroll
            for (int j = 0; j < 16; ++j) u[j] *= s.of(base + e0 + (j << 7) + (x << 13));
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) q[(j << 7) + (x << 13)] = u[j] * scale;
    }
}

// Index bits [14, 14 + B), in place: the pass behind the tile kernel.  A block takes 2^B elements 2^14 apart x 2^(14 - B) side by side
// (B > 5: the top five bits, then the others, through shared memory) or a thread 2^B (B <= 5, in registers).  The distance is
// a constant here, so that an element's address is the thread's plus a constant: with the distance in a register (fwht_cols_kernel) the
// addresses were most of the instructions, 36.5 -> 25.6 us for 2^24 elements, a copy of which takes 28.1.
template <int B, bool SIGNS>
__global__ void __launch_bounds__(B > 5 ? RHT_THREADS : 256, 2) fwht_next_kernel(float *W, RhtSigns s, float scale)
{
    constexpr int LT = RHT_TILE_BITS;
    constexpr int64_t ST = (int64_t)1 << LT;
    const int t = threadIdx.x;
    auto sign = [&](int64_t at) { return SIGNS ? scale * __ldg(s.rows + (at >> s.ln)) : scale; };
    if constexpr (B <= 5) {
        const int64_t q = (int64_t)blockIdx.x * blockDim.x + t;
        const int64_t base = (q & (ST - 1)) | ((q >> LT) << (LT + B));
        float v[1 << B], *p = W + base;
#pragma unroll
        for (int j = 0; j < (1 << B); ++j) v[j] = p[j * ST];
        fwht_reg<B>(v);
        if (SIGNS) scale *= __ldg(s.cols + (base & (((int64_t)1 << s.ln) - 1)));
#pragma unroll
        for (int j = 0; j < (1 << B); ++j) p[j * ST] = v[j] * sign(base + j * ST);
    } else {
        constexpr int L = B - 5, LC = LT - B, C = 1 << LC, PITCH = (1 << (L + LC)) + 16;     // (see fwht_cols_kernel)
        extern __shared__ __align__(16) float tile[];
        const int cl = t & (C - 1), r = t >> LC;
        const int64_t base = (int64_t)(blockIdx.x & ((1 << B) - 1)) * C + ((int64_t)(blockIdx.x >> B) << (LT + B)) + cl;
        float v[32];
        const float *p = W + base + r * ST;
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = p[j * (ST << L)];
        fwht_reg<5>(v);
        float *p1 = tile + (r << LC) + cl;
#pragma unroll
        for (int j = 0; j < 32; ++j) p1[j * PITCH] = v[j];
        __syncthreads();
        if (SIGNS) scale *= __ldg(s.cols + (base & (((int64_t)1 << s.ln) - 1)));
#pragma unroll
        for (int q = 0; q < (32 >> L); ++q) {
            const int rh = r + (q << L);
            const int64_t at = base + (int64_t)rh * (ST << L);
            float u[1 << L], *o = W + at;
#pragma unroll
            for (int j = 0; j < (1 << L); ++j) u[j] = tile[rh * PITCH + (j << LC) + cl];
            fwht_reg<L>(u);
#pragma unroll
            for (int j = 0; j < (1 << L); ++j) o[j * ST] = u[j] * sign(at + j * ST);
        }
    }
}

// Row-index bits [o, o + B), in place: a block takes 2^B rows (2^o apart) x 2^LC columns.  B <= 5: in registers, a thread per column and row group;
// B > 5: the top five bits, then the others, through shared memory (2^(B - 5 + LC) threads, 512 when the matrix is wide enough).
// sign_mode 2: outputs times their signs.
template <int B>
__global__ void __launch_bounds__(B > 5 ? RHT_THREADS : 256, 2) fwht_cols_kernel(float *W, RhtSigns s, int o, int LC, float scale, int sign_mode)
{
    extern __shared__ __align__(16) float tile[];
    const int t = threadIdx.x, C = 1 << LC;
    const int cblocks = 1 << (s.ln - LC);
    const int c = (int)(blockIdx.x & (cblocks - 1)) * C + (t & (C - 1));
    if (B <= 5) {
        const int64_t g = ((int64_t)(blockIdx.x >> (s.ln - LC)) * blockDim.x + t) >> LC;      // row group
        const int64_t row0 = ((g >> o) << (o + B)) | (g & (((int64_t)1 << o) - 1));
        constexpr int N = B <= 5 ? B : 1;
        float v[1 << N];
        float *p = W + (row0 << s.ln) + c;
        const int64_t stride = (int64_t)1 << (o + s.ln);
#pragma unroll
        for (int j = 0; j < (1 << N); ++j) v[j] = p[j * stride];
        fwht_reg<N>(v);
        if (sign_mode == 2) scale *= __ldg(s.cols + c);
#pragma unroll
        for (int j = 0; j < (1 << N); ++j) p[j * stride] = v[j] * scale * (sign_mode == 2 ? __ldg(s.rows + row0 + ((int64_t)j << o)) : 1.f);
    } else {
        constexpr int L = B > 5 ? B - 5 : 1;                     // bits of the second pass
        const int64_t g = blockIdx.x >> (s.ln - LC);
        const int64_t row0 = ((g >> o) << (o + B)) | (g & (((int64_t)1 << o) - 1));
        const int r = t >> LC;                                   // 0 .. 2^L - 1
        const int64_t stride = (int64_t)1 << (o + s.ln);
        float v[32];
        {
            const float *p = W + ((row0 + ((int64_t)r << o)) << s.ln) + c;
            const int64_t stride_hi = stride << L;
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = p[j * stride_hi];
        }
        fwht_reg<5>(v);
        if (sign_mode == 2) scale *= __ldg(s.cols + c);
        const int cl = t & (C - 1);
        // element (row, column) at (row >> L) * pitch + ((row & (2^L - 1)) << LC) + column; sixteen floats of padding in the pitch put the
        // second pass's two rows of a warp on different banks
        const int pitch = (1 << (L + LC)) + 16;
        float *p1 = tile + (r << LC) + cl;
#pragma unroll
        for (int j = 0; j < 32; ++j) p1[j * pitch] = v[j];
        __syncthreads();
#pragma unroll 1
        for (int q = 0; q < (32 >> L); ++q) {
            const int rh = r + (q << L);
            float u[1 << L];
#pragma unroll
            for (int j = 0; j < (1 << L); ++j) u[j] = tile[rh * pitch + (j << LC) + cl];
            fwht_reg<L>(u);
            const int64_t row = row0 + ((int64_t)(rh << L) << o);
            float *p = W + (row << s.ln) + c;
#pragma unroll
            for (int j = 0; j < (1 << L); ++j) p[j * stride] = u[j] * scale * (sign_mode == 2 ? __ldg(s.rows + row + ((int64_t)j << o)) : 1.f);
        }
    }
}

// scales[g] = sqrt(mean of the 16 squares of group g); out = W / scale (0 where the group is all zero).  Four lanes per group,
// one float4 each: a warp reads and writes 512 consecutive bytes.
__global__ void __launch_bounds__(256) group_scale_kernel(const float *W, float *scales, float *out, int64_t groups)
{
    const int64_t quads = 4 * groups, step = (int64_t)gridDim.x * blockDim.x;
    const uint64_t policy = rht_stream_policy();
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < quads; q += step) {      // (whole groups of lanes: quads and step are multiples of 4)
        const float4 v = rht_stream4(reinterpret_cast<const float4 *>(W) + q, policy);
        const unsigned mask = __activemask();
        float ss = v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
        ss += __shfl_xor_sync(mask, ss, 1);
        ss += __shfl_xor_sync(mask, ss, 2);
        const float sc = sqrtf(ss * (1.f / 16.f));
        const float inv = sc > 0.f ? 1.f / sc : 0.f;
        if ((q & 3) == 0) scales[q >> 2] = sc;
        reinterpret_cast<float4 *>(out)[q] = make_float4(v.x * inv, v.y * inv, v.z * inv, v.w * inv);
    }
}

// out = W_scaled * scale of its group
__global__ void __launch_bounds__(256) group_unscale_kernel(const float *Ws, const float *scales, float *out, int64_t groups)
{
    const int64_t quads = 4 * groups, step = (int64_t)gridDim.x * blockDim.x;
    const uint64_t policy = rht_stream_policy();
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < quads; q += step) {
        const float4 v = rht_stream4(reinterpret_cast<const float4 *>(Ws) + q, policy);
        const float sc = __ldg(scales + (q >> 2));
        reinterpret_cast<float4 *>(out)[q] = make_float4(v.x * sc, v.y * sc, v.z * sc, v.w * sc);
    }
}

}  // namespace bcjr
