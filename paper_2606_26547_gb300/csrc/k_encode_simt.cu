// K0: random-projection encoding on CUDA cores (FFMA), fused with
// sign binarisation and bit packing (Listing 1 __hetero_hdc_matmul followed
// by Automatic Binarization, Sec. 4.2).
//
// s[i][k] = sum_f X[i][f] * Bq[k][f] in FP32; bit = s < 0 (sign(0) = +1);
// 32 consecutive dims per word.  With FP32 inputs this is the plain exact
// form of the method; with BF16/FP8 inputs the products are exact in FP32,
// which gives a CUDA-core cross-check of the tensor-core encoder.
//
// Tiling: 128 queries x 64 * CG dims per block (CG = 4, or 2 with few features or where that leaves
// SMs idle), K slabs of 16, 256 threads with 8 x 4 * CG outputs each (rows
// ty*4+{0..3} and 64+ty*4+{0..3}, columns tx*4+{0..3} of every 64),
// double-buffered shared memory with register prefetch.
//
// Bound by the FP32 pipe (128 multiply-adds per clock per SM, 74.8 TFLOP/s
// measured).  Two columns a packed multiply-add (fma.rn.f32x2): the same
// rounding and order per output as one by one, in half the instructions, so
// that the loads issue beside the pipe's work; 8 x 16 outputs a thread take six
// 16-byte fragment loads per 128 multiply-adds (8 x 8: four per 64).  Query rows
// that are not 16-byte aligned (F % 4 != 0) are read a float per lane in 64-byte
// runs: the per-row alignment test ran the vector and the scalar loads of every
// warp.  10,000 rows to 10,000 dims: F = 784 3,121 -> 2,716 us (57.7 TFLOP/s),
// F = 561 2,427 -> 2,072 us.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include "hdc_internal.cuh"

namespace hdc {
namespace {

constexpr int BM = 128, BK = 16, LDS = BM + 4;
template <int CG>
constexpr int simt_smem() { return 2 * BK * (LDS + 64 * CG + 4) * 4; }

__device__ __forceinline__ void cvt4(const float *p, float *v)
{
    float4 t = *reinterpret_cast<const float4 *>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void cvt4(const __nv_bfloat16 *p, float *v)
{
    uint2 t = *reinterpret_cast<const uint2 *>(p);
    __nv_bfloat162 a = *reinterpret_cast<__nv_bfloat162 *>(&t.x), b = *reinterpret_cast<__nv_bfloat162 *>(&t.y);
    float2 fa = __bfloat1622float2(a), fb = __bfloat1622float2(b);
    v[0] = fa.x; v[1] = fa.y; v[2] = fb.x; v[3] = fb.y;
}
__device__ __forceinline__ float fp8_to_f(uint8_t b)
{
    __half_raw h = __nv_cvt_fp8_to_halfraw((__nv_fp8_storage_t)b, __NV_E4M3);
    return __half2float(__half(h));
}
__device__ __forceinline__ void cvt4(const uint8_t *p, float *v)
{
    uint32_t t = *reinterpret_cast<const uint32_t *>(p);
#pragma unroll
    for (int j = 0; j < 4; j++) v[j] = fp8_to_f((uint8_t)(t >> (8 * j)));
}
__device__ __forceinline__ float cvt1(const float *p) { return *p; }
__device__ __forceinline__ float cvt1(const __nv_bfloat16 *p) { return __bfloat162float(*p); }
__device__ __forceinline__ float cvt1(const uint8_t *p) { return fp8_to_f(*p); }

// Four consecutive elements [f, f+4) of a row, zero outside [0, F) or for an
// invalid row; vector load when the four are in range and aligned.
template <typename T>
__device__ __forceinline__ void load4(const T *row, bool valid, int f, int F, float *v)
{
    if (valid && f + 3 < F && (reinterpret_cast<uintptr_t>(row + f) % (4 * sizeof(T))) == 0) {
        cvt4(row + f, v);
        return;
    }
#pragma unroll
    for (int j = 0; j < 4; j++) v[j] = (valid && f + j < F) ? cvt1(row + f + j) : 0.f;
}

// acc + (a, a) * (b.x, b.y): two multiply-adds, each rounded once.
__device__ __forceinline__ void fma2(float2 &acc, float a, float2 b)
{
    asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %2};\n\tmov.b64 y, {%3, %4};\n\tmov.b64 z, {%0, %1};\n\t"
        "fma.rn.f32x2 z, x, y, z;\n\tmov.b64 {%0, %1}, z;\n\t}"
        : "+f"(acc.x), "+f"(acc.y)
        : "f"(a), "f"(b.x), "f"(b.y));
}

// VEC: the rows of X are 16-byte aligned (or T is a quantised, padded type).
template <typename T, bool VEC, int CG>
__global__ void __launch_bounds__(256, CG == 4 ? 1 : 2) encode_simt_kernel(const T *__restrict__ X, int64_t ldx, int64_t N, int F,
                                                             const T *__restrict__ B, int ldb, int Dk,
                                                             const float *__restrict__ sx, const float *__restrict__ sb,
                                                             uint32_t *__restrict__ H, int W, float *__restrict__ scores)
{
    constexpr int BN = 64 * CG, LDB = BN + 4;
    extern __shared__ __align__(16) float sm[];
    float(*As)[BK][LDS] = reinterpret_cast<float(*)[BK][LDS]>(sm);
    float(*Bs)[BK][LDB] = reinterpret_cast<float(*)[BK][LDB]>(sm + 2 * BK * LDS);
    // a warp's threads as 4 x 8 (rows x columns): its fragment loads touch 64
    // and 128 bytes of a slab row
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tx = (warp & 1) * 8 + (lane & 7), ty = (warp >> 1) * 4 + (lane >> 3);
    const int ltx = tid & 15, lty = tid >> 4;   // loader of unaligned query rows
    const int64_t m0 = (int64_t)blockIdx.y * BM;
    const int n0 = blockIdx.x * BN;

    // loader mapping: rows lr and lr+64, k offset lk; unaligned query rows:
    // column ltx of rows lty, lty+16, ...
    const int lr = tid >> 2, lk = (tid & 3) * 4;
    const T *arow0 = X + (m0 + (VEC ? lr : lty)) * ldx, *arow1 = X + (m0 + lr + 64) * ldx;
    const bool av0 = m0 + lr < N, av1 = m0 + lr + 64 < N;
    const T *brow0 = B + (int64_t)(n0 + lr) * ldb;   // rows lr, lr + 64, ... of the tile

    float ra[8], rb[4 * CG];
    auto gload = [&](int k0) {
        if (VEC) {
            load4(arow0, av0, k0 + lk, F, ra);
            load4(arow1, av1, k0 + lk, F, ra + 4);
        } else {
            const bool kin = k0 + ltx < F;
#pragma unroll
            for (int i = 0; i < 8; i++) ra[i] = kin && m0 + lty + 16 * i < N ? cvt1(arow0 + (int64_t)(16 * i) * ldx + k0 + ltx) : 0.f;
        }
#pragma unroll
        for (int g = 0; g < CG; g++) load4(brow0 + (int64_t)(64 * g) * ldb, n0 + lr + 64 * g < Dk, k0 + lk, F, rb + 4 * g);
    };
    auto sstore = [&](int buf) {
        if (VEC) {
#pragma unroll
            for (int j = 0; j < 4; j++) {
                As[buf][lk + j][lr] = ra[j];
                As[buf][lk + j][lr + 64] = ra[4 + j];
            }
        } else {
#pragma unroll
            for (int i = 0; i < 8; i++) As[buf][ltx][lty + 16 * i] = ra[i];
        }
#pragma unroll
        for (int g = 0; g < CG; g++)
#pragma unroll
            for (int j = 0; j < 4; j++) Bs[buf][lk + j][lr + 64 * g] = rb[4 * g + j];
    };

    float2 acc2[8][2 * CG];
#pragma unroll
    for (int i = 0; i < 8; i++)
#pragma unroll
        for (int j = 0; j < 2 * CG; j++) acc2[i][j] = make_float2(0.f, 0.f);

    const int nk = (F + BK - 1) / BK;
    gload(0);
    sstore(0);
    __syncthreads();
    for (int kt = 0; kt < nk; kt++) {
        const int cur = kt & 1;
        if (kt + 1 < nk) gload((kt + 1) * BK);
#pragma unroll
        for (int kk = 0; kk < BK; kk++) {
            float a[8];
            float2 b[2 * CG];
            *reinterpret_cast<float4 *>(a) = *reinterpret_cast<const float4 *>(&As[cur][kk][ty * 4]);
            *reinterpret_cast<float4 *>(a + 4) = *reinterpret_cast<const float4 *>(&As[cur][kk][64 + ty * 4]);
#pragma unroll
            for (int g = 0; g < CG; g++)
                *reinterpret_cast<float4 *>(b + 2 * g) = *reinterpret_cast<const float4 *>(&Bs[cur][kk][64 * g + tx * 4]);
#pragma unroll
            for (int j = 0; j < 2 * CG; j++)   // the column pair reused over the rows: 4 % faster than the other way
#pragma unroll
                for (int i = 0; i < 8; i++) fma2(acc2[i][j], a[i], b[j]);
        }
        if (kt + 1 < nk) sstore(cur ^ 1);
        __syncthreads();
    }
    auto acc = [&](int i, int j) { return j & 1 ? acc2[i][j >> 1].y : acc2[i][j >> 1].x; };

    // ---- epilogue: optional projections, then sign -> pack ---------------
#pragma unroll
    for (int i = 0; i < 8; i++) {
        const int64_t row = m0 + (i < 4 ? ty * 4 + i : 64 + ty * 4 + i - 4);
        if (scores != nullptr && row < N) {
            const float rs = sx ? sx[row] : 1.f;
#pragma unroll
            for (int j = 0; j < 4 * CG; j++) {
                const int col = n0 + j / 4 * 64 + tx * 4 + j % 4;
                if (col < Dk) scores[row * Dk + col] = acc(i, j) * rs * (sb ? sb[col] : 1.f);
            }
        }
#pragma unroll
        for (int h = 0; h < CG; h++) {
            uint32_t nib = 0;
#pragma unroll
            for (int j = 0; j < 4; j++) nib |= (acc(i, h * 4 + j) < 0.f ? 1u : 0u) << j;
            uint32_t v = nib << (4 * (tx & 7));
            v |= __shfl_xor_sync(0xffffffffu, v, 1);
            v |= __shfl_xor_sync(0xffffffffu, v, 2);
            v |= __shfl_xor_sync(0xffffffffu, v, 4);
            if ((tx & 7) == 0 && row < N) {
                const int word = n0 / 32 + h * 2 + (tx >> 3);
                if (word < W) H[row * W + word] = v;
            }
        }
    }
}

template <typename T, bool VEC, int CG>
cudaError_t launch_simt(const void *X, int64_t ldx, int64_t n, int F, const void *Bq, int ldb, int Dk, const float *sx,
                        const float *sb, uint32_t *H, int W, float *scores, cudaStream_t st)
{
    auto k = encode_simt_kernel<T, VEC, CG>;
    constexpr int smem = simt_smem<CG>();
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
    }
    const dim3 grid((Dk + 64 * CG - 1) / (64 * CG), (unsigned)((n + BM - 1) / BM));
    k<<<grid, 256, smem, st>>>((const T *)X, ldx, n, F, (const T *)Bq, ldb, Dk, sx, sb, H, W, scores);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_encode_simt(const void *X, int64_t ldx, int64_t N, int F, const void *Bq, int ldb, int Dk, int enc,
                               const float *sx, const float *sb, uint32_t *H, int W, float *scores, cudaStream_t st)
{
    const int64_t chunk = (int64_t)65535 * BM;  // grid.y limit per launch
    const int es = esize_for(enc);
    for (int64_t off = 0; off < N; off += chunk) {
        const int64_t n = N - off < chunk ? N - off : chunk;
        const char *Xc = (const char *)X + off * ldx * es;
        const float *sxc = sx ? sx + off : nullptr;
        uint32_t *Hc = H + off * W;
        float *sc = scores ? scores + off * Dk : nullptr;
        // Waves of the wide tile (one block per SM) against the narrow one's (two,
        // each at half the rate; a lone one at the full rate), in 128 x 128
        // tiles; the wide one runs ~10 % faster where both fill the chip
        // (5,000 x 617 x 2,048, 2.1 waves of the wide tile: 284 us narrow, 338 us wide).
        // Not below 16 K slabs: a block's own ends, the stores of its projections
        // above all, pass beside another block's multiply-adds on the narrow tile
        // only (42,413 x 10 x 1,685 with projections: 136 us narrow, 177 wide; x 64:
        // 252 / 302; without, x 16: 64 / 78; from 300 features 0.9 .. 1.04).
        const int64_t mt = (n + BM - 1) / BM, bw = mt * ((Dk + 255) / 256), bn = mt * ((Dk + 127) / 128);
        const int64_t rem = bn % 304, cn = bn / 304 * 2 + (rem > 152 ? 2 : rem > 0 ? 1 : 0);
        const bool wide = F >= 16 * BK && (bw + 151) / 152 * 18 < cn * 10;
        cudaError_t e;
#define HDC_SIMT(T, V) \
    (wide ? launch_simt<T, V, 4>(Xc, ldx, n, F, Bq, ldb, Dk, sxc, sb, Hc, W, sc, st) \
          : launch_simt<T, V, 2>(Xc, ldx, n, F, Bq, ldb, Dk, sxc, sb, Hc, W, sc, st))
        switch (enc) {
        case HDC_ENC_FP32:
            e = ldx % 4 == 0 && (uintptr_t)Xc % 16 == 0 ? HDC_SIMT(float, true) : HDC_SIMT(float, false);
            break;
        case HDC_ENC_BF16: e = HDC_SIMT(__nv_bfloat16, true); break;
        default: e = HDC_SIMT(uint8_t, true);
        }
#undef HDC_SIMT
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace hdc
