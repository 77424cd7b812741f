// Packed +-1 rows against small-integer class rows on the tensor cores (up to
// 256 class rows).  What the dot products are for (FIN):
//   HP_HAMMING  the Hamming arg-min of packed binary hypervectors (Sec. 4.1
//               Hamming distance and arg-min primitives);
//   HP_COSINE   the cosine arg-max against b-bit class hypervectors (Sec. 4.2
//               Algorithmic Choice);
//   HP_SWEEP    the arg-max of every (class width, perforation) configuration
//               of a trained model, its correct predictions counted;
//   HP_FEW      HP_HAMMING with distances of few rows of a class number that is
//               no multiple of four, which are not worth staging.
// A b-bit class value is P signed base-16 digits (1 for up to 4 bits, 2 for 8,
// 8 for 32), each a class row of its own that E4M3 holds exactly; the digits'
// dot products, exact in FP32 (at most 8 * 131,072), are put together as
// integers.
//
// For +-1 vectors over the kept dims K, Hamming(q, c) = (|K| - q.c) / 2, and
// q.c is an exact integer in FP32.  The packed words are expanded to E4M3
// bytes: +1.0 (0x38) for bit 0, -1.0 (0xB8) for bit 1.  The dims of a 32-dim
// word are taken in the order j + 8k (j = 0..7 the 32-bit group, k = 0..3 its
// byte), the same for both operands, so that a group of four dims is
//   ((w << (7 - j)) & 0x80808080) | 0x38383838
// -- one shift and one logic operation, no bit transposition.  Only the class
// bytes carry the kept dims (0 outside K and past D): the query bytes need no
// mask.  Then
//   D2 += Qtile . Ctile^T     (M 128 queries, N = R class rows, K = 32 bytes)
// accumulates over the row in tensor memory.
//
// One CTA per SM, persistent over units of MT x 128 query rows (MT = 2 up to
// 128 class rows: the class bytes, R x D per unit, are the larger stream).
// Roles (27 warps):
//   warps 0-15  expand: a thread takes its row's 128 dims of an atom (MT = 2:
//               every second atom; MT = 1: every fourth) from the staged query words and writes them into its own
//               TMEM lane (tcgen05.st): operand A of the MMAs, a ring of NAB
//               atom buffers.  The bytes are formed before the wait for the
//               buffer, so only the store and the MMAs are in its chain;
//   warps 16-23 epilogue: D2 -> distances and arg-min, while the next unit's
//               atoms accumulate into the other D2 (R <= 64); distances leave
//               through shared memory as runs of a row;
//   warp 24     TMA producer of the packed query words, 1,024 dims x MT x 128
//               rows per copy (whole 128-byte lines), a ring of HP_QB chunks;
//   warp 25     PRE: TMA producer of the class bytes (atoms of R rows x 128
//               dims) into a ring of p.nbs slots;
//   warp 26     MMA issuer.
// PRE: the class rows come already expanded (R rows of bytes in this dim order:
// class_bytes_kernel's in the caller's workspace, a model's digit rows, or the
// sweep's).  Without it the expanding
// warps also expand the class words of every tile into two shared-memory
// buffers.
//
// Split rows: a batch of few units is given to clusters of p.S CTAs, each
// accumulating a contiguous part of the dims; the partial D2 are exchanged
// through distributed shared memory and the row groups of the unit are
// finished by the ranks in turn.
//
// TMEM (512 columns): D2 in columns 0..255 (MT x RS columns a buffer, RS = R
// rounded up to 32), the NAB query buffers of MT x 32 columns from 256.
// Every barrier wait is bounded as in the encoder.  The cluster barriers of a split
// row are not: every thread of every rank reaches both, an aborted one too, and
// the ranks of a cluster run together.
//
// Bound by an atom's barrier, store and MMA-issue latencies one after the other
// (~420 cycles for 128 dims; no pipe is full).  The forms' times: launch_hamming_packed.
#pragma once
#include "tc_hamming.cuh"

namespace hdc {
namespace tc {

constexpr int HP_EXPW = 16;                    // expanding warps (0-15)
constexpr int HP_EPI0 = HP_EXPW;               // first of the eight epilogue warps
constexpr int HP_QPROD = HP_EXPW + 8, HP_BPROD = HP_EXPW + 9, HP_ISSUER = HP_EXPW + 10;
constexpr int HP_THREADS = (HP_EXPW + 11) * 32;
constexpr int HP_CMAX = 256;
constexpr int HP_MAX_W = 4096;                 // words of a packed row (D <= 131072)
constexpr int HP_QB = 3;                       // query chunks in the ring
constexpr int HP_CHUNK = 4;                    // 256-dim tiles per query chunk (128 bytes of a row)
constexpr int HP_NBS_MAX = 16;                 // most class-atom slots
constexpr int HP_SMAX = 8;                     // most CTAs a unit's dims are split over
constexpr int HP_HAMMING = 0, HP_COSINE = 1, HP_SWEEP = 2, HP_FEW = 3;
constexpr int HP_MAXCFG = HDC_SWEEP_MAX_STRIDES * HDC_SWEEP_MAX_BITS;
constexpr uint32_t HP_ACOL = 256;              // first TMEM column of the query buffers
constexpr int HP_NAB_MAX = 8;                  // query-atom buffers: 4, or 8 with MT = 1 and PRE
__host__ __device__ constexpr int hp_nab(int mt, bool pre) { return mt == 1 && pre ? 8 : 4; }
// qfull[QB], qempty[QB], bfull[NBS], bempty[NBS], afull[NAB], aempty[NAB], d2full[2], d2empty[2], done
constexpr int HP_NUM_BARS = 2 * HP_QB + 2 * HP_NBS_MAX + 2 * HP_NAB_MAX + 5;
constexpr int HP_OUT = 32 * 33 * 4;            // an epilogue warp's 32 x 32 distances, padded rows
// epilogue staging, barriers, TMEM slot, abort flag
__host__ __device__ constexpr int hp_tail(int mt) { return 4 * mt * HP_OUT + HP_NUM_BARS * 8 + 16; }

__host__ __device__ constexpr int hp_q_bytes(int mt) { return HP_QB * mt * 128 * 128; }

struct HPParams {
    const uint32_t *cls;     // C x W packed class hypervectors (not PRE)
    int64_t N;
    int W, C, R, nt;         // R: C rounded up to 16; nt: 256-dim tiles = ceil(W / 8)
    int nbs;                 // PRE: class-atom slots
    int S;                   // CTAs of a cluster that share a unit's dims
    int64_t D, s0, e0, stride;   // dims of the rows; kept dims s0 + k*stride < e0 (stride 1, [0, D) if none)
    int kept;                // |K|
    int32_t *labels, *dists;
    // HP_COSINE: digits of a class value, class norms, optional scores (N x C)
    int P;
    const double *cnorm;
    double *scores;
    // HP_SWEEP: ncfg configurations of C classes; configuration i owns the
    // class rows [cfg_col, cfg_col + C * cfg_p), class by class, its digits
    // side by side (cfg_p 0: one sign row, Hamming), and writes output entry
    // cfg_k; sumsq[cfg_k * C + c]: sum of the squared class values it keeps
    int ncfg;
    uint8_t cfg_p[HP_MAXCFG], cfg_k[HP_MAXCFG];
    uint16_t cfg_col[HP_MAXCFG];
    int64_t ldl;             // labels from one output entry to the next
    const long long *sumsq;
    const int32_t *y;
    int32_t *correct;
};

// Four dims j, j + 8, j + 16, j + 24 of a packed word as E4M3 +-1 bytes.
__device__ __forceinline__ uint32_t hp_signs(uint32_t w, int j) { return ((w << (7 - j)) & 0x80808080u) | 0x38383838u; }
// The same four dims of a mask word as bytes 0xFF (set) or 0.
__device__ __forceinline__ uint32_t hp_mask(uint32_t m, int j) { return ((m >> j) & 0x01010101u) * 0xFFu; }

// Kept dims of word w: s0, s0 + stride, ... below min(e0, D).
__host__ __device__ __forceinline__ uint32_t hp_word_mask(int64_t w, int64_t D, int64_t s0, int64_t e0, int64_t stride)
{
    const int64_t base = w * 32, end = e0 < D ? e0 : D;
    const int64_t lo = s0 > base ? s0 : base, hi = end < base + 32 ? end : base + 32;
    if (lo >= hi) return 0;
    if (stride == 1) {
        const int a = (int)(lo - base), b = (int)(hi - base);
        return (b == 32 ? 0xffffffffu : ((1u << b) - 1u)) & ~((1u << a) - 1u);
    }
    uint32_t m = 0;
    const int64_t r0 = (lo - s0) % stride;
    for (int64_t d = r0 ? lo + (stride - r0) : lo; d < hi; d += stride) m |= 1u << (d - base);
    return m;
}

// Thirty-two 32-bit TMEM columns of this thread's lane.
__device__ __forceinline__ void hp_tmem_st32(uint32_t taddr, const uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
        "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]),
        "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),
        "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}

// NW words of class row r into its 128-byte row of a K atom (128-byte
// swizzle), from 16-byte piece `p0` on; zero outside the mask words.  A class
// row past C has zero words: its products are never read.
template <int NW>
__device__ __forceinline__ void hp_expand_row(uint8_t *atom, int r, int p0, const uint4 w, const uint4 m)
{
    uint8_t *row = atom + r * 128;
    const uint32_t ws[4] = {w.x, w.y, w.z, w.w}, ms[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
    for (int i = 0; i < NW; i++) {
        uint32_t b[8];
#pragma unroll
        for (int j = 0; j < 8; j++) b[j] = hp_signs(ws[i], j) & hp_mask(ms[i], j);
        *reinterpret_cast<uint4 *>(row + (((p0 + 2 * i) ^ (r & 7)) * 16)) = make_uint4(b[0], b[1], b[2], b[3]);
        *reinterpret_cast<uint4 *>(row + (((p0 + 2 * i + 1) ^ (r & 7)) * 16)) = make_uint4(b[4], b[5], b[6], b[7]);
    }
}

// Eight 32-bit TMEM columns of this thread's lane.
__device__ __forceinline__ void hp_tmem_ld8(uint32_t taddr, uint32_t (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7])
                 :
                 : "memory");
}

// Value of P digit dot products (exact integers): the digits' weights are the
// powers of 16.
template <int P>
__device__ __forceinline__ long long hp_digits(const uint32_t *v)
{
    long long d = 0;
#pragma unroll
    for (int q = P - 1; q >= 0; q--) d = d * 16 + (long long)(int)__uint_as_float(v[q]);
    return d;
}

// The same rounded once to FP32: exact for P <= 2 (below 2^24).  Eight digits
// may cancel, so they are put together as integers first.
template <int P>
__device__ __forceinline__ float hp_digits_f(const uint32_t *v)
{
    if (P == 1) return __uint_as_float(v[0]);
    if (P == 2) return fmaf(__uint_as_float(v[1]), 16.f, __uint_as_float(v[0]));
    return (float)hp_digits<P>(v);
}

// a / b correctly rounded from y = 1 / b correctly rounded (0 for b = 0, which
// gives 0): P. Markstein, "Computation of elementary functions on the IBM RISC
// System/6000 processor", IBM J. Res. Dev. 34(1), 1990: one step makes the
// quotient faithful, the next one correct.  Integers a and norms b: no
// overflow, no subnormals.
__device__ __forceinline__ double hp_div(double a, double b, double y)
{
    double q = a * y;
    q = fma(fma(-q, b, a), y, q);
    return fma(fma(-q, b, a), y, q);
}

__device__ __forceinline__ void hp_cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// A 32-bit word at this CTA's shared address `a`, in the cluster's CTA `rank`.
__device__ __forceinline__ float hp_ld_cluster(uint32_t a, uint32_t rank)
{
    float v;
    asm volatile("{\n\t.reg .b32 r;\n\tmapa.shared::cluster.u32 r, %1, %2;\n\tld.shared::cluster.f32 %0, [r];\n\t}"
                 : "=f"(v)
                 : "r"(a), "r"(rank));
    return v;
}

template <int V>
struct HpInt {
    static constexpr int value = V;
};

template <int MT, bool PRE, int FIN = HP_HAMMING>
__global__ void __launch_bounds__(HP_THREADS, 1)
    tc_hamming_packed_kernel(const HPParams p, const __grid_constant__ CUtensorMap tmQ,
                             const __grid_constant__ CUtensorMap tmC)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    constexpr int UROWS = MT * BM;                               // query rows of a unit
    constexpr int QCH = UROWS * 128;                             // bytes of a query chunk
    uint8_t *sQ = smem;
    constexpr int NAB = hp_nab(MT, PRE);
    constexpr bool HAM = FIN == HP_HAMMING || FIN == HP_FEW;
    uint8_t *sB = smem + hp_q_bytes(MT);                         // class atoms: nbs, or one per query buffer
    const int atom_bytes = p.R * 128;
    int32_t *s_out = reinterpret_cast<int32_t *>(sB + (size_t)(PRE ? p.nbs : NAB) * atom_bytes);   // 4 * MT x HP_OUT
    uint64_t *bars = reinterpret_cast<uint64_t *>(s_out + 4 * MT * (HP_OUT / 4));
    uint32_t *smask = reinterpret_cast<uint32_t *>(bars + HP_NUM_BARS + 1);   // W words (not PRE)
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + HP_NUM_BARS);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    auto qfull = [&](int b) { return su32(bars + b); };
    auto qempty = [&](int b) { return su32(bars + HP_QB + b); };
    auto bfull = [&](int b) { return su32(bars + 2 * HP_QB + b); };
    auto bempty = [&](int b) { return su32(bars + 2 * HP_QB + HP_NBS_MAX + b); };
    constexpr int X = 2 * HP_QB + 2 * HP_NBS_MAX;
    auto afull = [&](int b) { return su32(bars + X + b); };
    auto aempty = [&](int b) { return su32(bars + X + HP_NAB_MAX + b); };
    auto d2full = [&](int b) { return su32(bars + X + 2 * HP_NAB_MAX + b); };
    auto d2empty = [&](int b) { return su32(bars + X + 2 * HP_NAB_MAX + 2 + b); };
    const uint32_t done_bar = su32(bars + X + 2 * HP_NAB_MAX + 4);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int RS = (p.R + 31) & ~31;                 // D2 columns of one 128-row tile
    const int ND2 = MT * RS <= 128 ? 2 : 1;          // D2 buffers
    const int64_t units = (p.N + UROWS - 1) / UROWS;
    const int S = p.S;
    const int rank = S > 1 ? (int)(blockIdx.x % S) : 0;
    const int64_t u0 = blockIdx.x / S, ustep = gridDim.x / S;
    const int chunks = (p.nt + HP_CHUNK - 1) / HP_CHUNK;
    const int ch0 = chunks * rank / S, ch1 = chunks * (rank + 1) / S;   // this rank's query chunks
    auto chunk_atoms = [&](int ch) { return 2 * min(HP_CHUNK, p.nt - ch * HP_CHUNK); };

    if (tid == 0) {
        for (int b = 0; b < HP_QB; b++) {
            mbar_init(qfull(b), 1);
            mbar_init(qempty(b), HP_EXPW);
        }
        for (int b = 0; b < HP_NBS_MAX; b++) {
            mbar_init(bfull(b), 1);
            mbar_init(bempty(b), 1);
        }
        for (int b = 0; b < NAB; b++) {
            mbar_init(afull(b), 4 * MT);
            mbar_init(aempty(b), 1);
        }
        for (int b = 0; b < 2; b++) {
            mbar_init(d2full(b), 1);
            mbar_init(d2empty(b), 4 * MT);
        }
        mbar_init(done_bar, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    grid_wait();
    // class norms and their reciprocals, 0 for a zero norm (cosine, sweep: no
    // distances are staged there)
    double *s_norm = reinterpret_cast<double *>(s_out), *s_rinv = s_norm + HP_CMAX;
    float *s_rinvf = reinterpret_cast<float *>(s_rinv + HP_CMAX);   // (narrowing takes the FP64 pipe: once here)
    if (!HAM)
        for (int i = tid; i < (FIN == HP_SWEEP ? p.ncfg : 1) * p.C; i += HP_THREADS) {
            const int f = FIN == HP_SWEEP ? i / p.C : 0;
            const double n = FIN == HP_COSINE ? p.cnorm[i] : sqrt((double)p.sumsq[(int64_t)p.cfg_k[f] * p.C + i % p.C]);
            s_norm[i] = n;
            const double y = n == 0.0 ? 0.0 : 1.0 / n;
            s_rinv[i] = y;
            s_rinvf[i] = (float)y;
        }
    if (!PRE)
        for (int w = tid; w < p.W; w += HP_THREADS) smask[w] = hp_word_mask(w, p.D, p.s0, p.e0, p.stride);
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_slot)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    // Distances and arg-min of the 32 rows from `row0` on (this lane's is
    // row0 + lane) from their R dot products, read 32 columns at a time by
    // cols(j, v); `out`: the warp's staging for the distances.
    auto finish = [&](int64_t row0, int32_t *out, auto cols) {
        int best = 0;
        float bd = -3.0e38f;   // largest dot = smallest distance; ascending c: lowest class on ties
        const bool vec = p.C % 4 == 0 && (reinterpret_cast<uintptr_t>(p.dists) & 15) == 0;
        const int nrow = (int)min((int64_t)32, p.N - row0);   // rows of this warp below N (may be <= 0)
        for (int j = 0; j * 32 < p.R; j++) {
            uint32_t v[32];
            cols(j, v);
            const int nc = min(32, p.C - j * 32);
#pragma unroll
            for (int i = 0; i < 32; i++) {
                const float d = __uint_as_float(v[i]);
                if (i < nc && d > bd) { bd = d; best = j * 32 + i; }
            }
            if (p.dists) {
#pragma unroll
                for (int i = 0; i < 32; i++) v[i] = (uint32_t)((p.kept - (int)__uint_as_float(v[i])) / 2);
                if (vec) {   // 16 bytes a store: 10^5 x 256 classes 23 us of distances (41 us staged)
                    int32_t *o = p.dists + (row0 + lane) * p.C + j * 32;
#pragma unroll
                    for (int i = 0; i < 32; i += 4)
                        if (i < nc && lane < nrow)
                            *reinterpret_cast<uint4 *>(o + i) = make_uint4(v[i], v[i + 1], v[i + 2], v[i + 3]);
                } else if (FIN == HP_FEW) {   // single words: one row of 255 classes 10 us (16 staged)
                    int32_t *o = p.dists + (row0 + lane) * p.C + j * 32;
#pragma unroll
                    for (int i = 0; i < 32; i++)
                        if (i < nc && lane < nrow) o[i] = (int32_t)v[i];
                } else {     // 10^6 x 33 classes: 44 us (125 us of single words)
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < 32; i++)
                        if (i < nc) out[lane * 33 + i] = (int32_t)v[i];
                    __syncwarp();
                    if (nc <= 2) {   // a lane its own row (10^6 x 128 dims x 33: 112 us by columns, 91 so)
                        int32_t *o = p.dists + (row0 + lane) * p.C + j * 32;
                        for (int i = 0; lane < nrow && i < nc; i++) o[i] = out[lane * 33 + i];
                        continue;
                    }
                    int32_t *o = p.dists + row0 * p.C + j * 32 + lane;
                    if (lane < nc)
#pragma unroll 8
                        for (int r = 0; r < 32; r++)
                            if (r < nrow) o[(int64_t)r * p.C] = out[r * 33 + lane];
                }
            }
        }
        if (lane < nrow) p.labels[row0 + lane] = best;
    };

    // Cosine arg-max of this lane's row from its C * P digit dot products,
    // read eight columns at a time by cols8(col, v).  The score is dot / norm
    // in FP64, lowest class first, as in the general kernel.  FP64 runs at a
    // few operations per clock per SM here, so the arg-max alone is taken in
    // FP32 (dot, 1 / norm and their product each rounded: within 2^-22 of the
    // score) and only classes within 2^-20 of the largest are compared in FP64:
    // a class below that cannot reach it.  With FP64 divisions for all, the
    // sweep's epilogue took 75 of its 86 us.
    auto arg_max = [&](int64_t row, bool valid, int col, int f0, double *scores, auto digits, auto cols8) {
        constexpr int P = decltype(digits)::value, CPL = 8 / P;   // classes a load
        int best = 0;
        if (scores) {
            double bs = 0.0;
            for (int c0 = 0; c0 < p.C; c0 += CPL) {
                uint32_t v[8];
                cols8(col + c0 * P, v);
#pragma unroll
                for (int i = 0; i < CPL; i++) {
                    const int c = c0 + i;
                    if (c < p.C) {
                        const double sc = hp_div((double)(int)hp_digits<P>(v + i * P), s_norm[f0 + c], s_rinv[f0 + c]);
                        if (valid) scores[row * p.C + c] = sc;
                        if (c == 0 || sc > bs) { bs = sc; best = c; }
                    }
                }
            }
            return best;
        }
        float top = -3.0e38f;
        int near_top = 0;   // classes that may reach the largest score
        for (int pass = 0; pass < 2; pass++) {
            const float lim = top - fabsf(top) * 0x1p-20f;
            for (int c0 = 0; c0 < p.C; c0 += CPL) {
                uint32_t v[8];
                cols8(col + c0 * P, v);
#pragma unroll
                for (int i = 0; i < CPL; i++) {
                    const int c = c0 + i;
                    if (c >= p.C) continue;
                    const float sc = hp_digits_f<P>(v + i * P) * s_rinvf[f0 + c];
                    if (pass == 0) {
                        top = fmaxf(top, sc);
                    } else if (sc >= lim) {
                        if (near_top++ == 0) best = c;
                    }
                }
            }
        }
        if (__any_sync(0xffffffffu, near_top > 1)) {   // a near tie in this warp: those rows again in FP64
            const float lim = top - fabsf(top) * 0x1p-20f;
            double bs = 0.0;
            bool first = true;
            for (int c0 = 0; c0 < p.C; c0 += CPL) {
                uint32_t v[8];
                cols8(col + c0 * P, v);
#pragma unroll
                for (int i = 0; i < CPL; i++) {
                    const int c = c0 + i;
                    if (c >= p.C) continue;
                    const long long d = hp_digits<P>(v + i * P);
                    if (hp_digits_f<P>(v + i * P) * s_rinvf[f0 + c] < lim) continue;
                    const double n = s_norm[f0 + c], sc = n == 0.0 ? 0.0 : (double)d / n;
                    if (first || sc > bs) { bs = sc; best = c; first = false; }
                }
            }
        }
        return best;
    };
    auto finish_scores = [&](int64_t row0, auto cols8) {
        const int64_t row = row0 + lane;
        const bool valid = row < p.N;
        if (FIN == HP_COSINE) {
            const int best = p.P == 1 ? arg_max(row, valid, 0, 0, p.scores, HpInt<1>(), cols8)
                                      : arg_max(row, valid, 0, 0, p.scores, HpInt<2>(), cols8);
            if (valid) p.labels[row] = best;
            return;
        }
        const int yv = valid ? p.y[row] : -1;
        for (int f = 0; f < p.ncfg; f++) {
            const int col = p.cfg_col[f];
            int best = 0;
            if (p.cfg_p[f] == 0) {   // signs: the largest dot product is the smallest distance
                float bd = -3.0e38f;
                for (int c0 = 0; c0 < p.C; c0 += 8) {
                    uint32_t v[8];
                    cols8(col + c0, v);
#pragma unroll
                    for (int i = 0; i < 8; i++)
                        if (c0 + i < p.C && __uint_as_float(v[i]) > bd) { bd = __uint_as_float(v[i]); best = c0 + i; }
                }
            } else if (p.cfg_p[f] == 1) {
                best = arg_max(row, valid, col, f * p.C, nullptr, HpInt<1>(), cols8);
            } else if (p.cfg_p[f] == 2) {
                best = arg_max(row, valid, col, f * p.C, nullptr, HpInt<2>(), cols8);
            } else {
                best = arg_max(row, valid, col, f * p.C, nullptr, HpInt<8>(), cols8);
            }
            if (valid && p.labels) p.labels[(int64_t)p.cfg_k[f] * p.ldl + row] = best;
            const unsigned hit = __ballot_sync(0xffffffffu, valid && best == yv);
            if (lane == 0 && hit) atomicAdd(p.correct + p.cfg_k[f], __popc(hit));
        }
    };

    if (warp == HP_ISSUER) {
        if (elect_one()) {  // ------------------------------ MMA issuer
            const uint32_t id = idesc_n<HDC_ENC_FP8_E4M3>(p.R);
            const uint64_t db0 = sdesc(su32(sB));
            int slot = 0, d2 = 0;
            uint32_t g = 0, bph = 0, d2ph[2] = {0, 0};   // g: atoms so far
            bool ab = false;
            for (int64_t u = u0; u < units && !ab; u += ustep) {
                if (!mbar_wait_fast(d2empty(d2), d2ph[d2] ^ 1, abort_flag)) { ab = true; break; }
                d2ph[d2] ^= 1;
                const uint32_t dcol = tmem + (uint32_t)(d2 * MT * RS);
                uint32_t accum = 0;
                for (int ch = ch0; ch < ch1 && !ab; ch++) {
                    const int na = chunk_atoms(ch);
                    for (int a = 0; a < na; a++, g++) {   // an atom: four 32-byte K steps of every query tile
                        const int buf = g % NAB;
                        if (!mbar_wait_fast(afull(buf), (g / NAB) & 1, abort_flag)) { ab = true; break; }
                        if (PRE && !mbar_wait_fast(bfull(slot), bph, abort_flag)) { ab = true; break; }
                        tc_fence_after();
                        const uint32_t acol = tmem + HP_ACOL + (uint32_t)(buf * MT * 32);
                        const uint64_t db = db0 + (uint64_t)(PRE ? slot : buf) * (uint64_t)(atom_bytes >> 4);
#pragma unroll
                        for (int m = 0; m < MT; m++)
#pragma unroll
                            for (int k = 0; k < 4; k++)
                                h_mma_ts_fp8(dcol + (uint32_t)(m * RS), acol + (uint32_t)(m * 32 + 8 * k), db + 2 * k, id,
                                             accum | (uint32_t)k);
                        accum = 1;
                        mma_commit(aempty(buf));
                        if (PRE) {
                            mma_commit(bempty(slot));
                            if (++slot == p.nbs) { slot = 0; bph ^= 1; }
                        }
                    }
                }
                if (ab) break;
                mma_commit(d2full(d2));
                if (++d2 == ND2) d2 = 0;
            }
            mma_commit(done_bar);   // all MMAs of this thread complete before TMEM is released
            const unsigned long long t0 = gtimer();
            while (!mbar_try(done_bar, 0) && gtimer() - t0 < 100000000ull) {}
        }
    } else if (warp == HP_QPROD || warp == HP_BPROD) {
        if ((PRE || warp == HP_QPROD) && elect_one()) {  // ---- TMA producers
            const bool isq = warp == HP_QPROD;
            const int nslots = isq ? HP_QB : p.nbs;
            int slot = 0;
            uint32_t ph = 0, issued = 0, par = 0;
            bool ab = false;
            for (int64_t u = u0; u < units && !ab; u += ustep)
                for (int ch = ch0; ch < ch1 && !ab; ch++) {
                    const int n = isq ? 1 : chunk_atoms(ch);   // a query chunk, or its class atoms
                    for (int a = 0; a < n; a++) {
                        const uint32_t fb = isq ? qfull(slot) : bfull(slot);
                        if (!mbar_wait_fast(isq ? qempty(slot) : bempty(slot), ph ^ 1, abort_flag)) { ab = true; break; }
                        if (isq) {
                            mbar_expect_tx(fb, QCH);
#pragma unroll
                            for (int m = 0; m < MT; m++)
                                tma_load_2d(su32(sQ + slot * QCH + m * (BM * 128)), &tmQ, ch * 32,
                                            (int)(u * UROWS + m * BM), fb);
                        } else {
                            mbar_expect_tx(fb, (uint32_t)atom_bytes);
                            tma_load_2d(su32(sB + slot * atom_bytes), &tmC, (ch * HP_CHUNK * 2 + a) * 128, 0, fb);
                        }
                        issued |= 1u << slot;
                        par = (par & ~(1u << slot)) | (ph << slot);
                        if (++slot == nslots) { slot = 0; ph ^= 1; }
                    }
                }
            if (ab)   // let this thread's copies land before the CTA exits
                for (int b = 0; b < nslots; b++)
                    if (issued >> b & 1) {
                        const unsigned long long t0 = gtimer();
                        while (!mbar_try(isq ? qfull(b) : bfull(b), par >> b & 1) && gtimer() - t0 < 100000000ull) {}
                    }
        }
    } else if (warp < HP_EPI0) {  // ---------------------- expanding warps
        const int urow = tid % UROWS;                           // row of the unit
        // every AS-th atom of the CTA, from number `grp` on: AS <= NAB, so a
        // buffer's phase is never two generations behind the one awaited
        constexpr int AS = HP_EXPW / (4 * MT);
        static_assert(AS <= NAB, "an expanding warp's next atom is at most one round of the buffers away");
        const uint32_t grp = (uint32_t)(warp / (4 * MT));
        const uint32_t tcol = tmem + ((uint32_t)((warp & 3) * 32) << 16) + HP_ACOL + (uint32_t)(urow / BM * 32);
        int qs = 0;
        uint32_t qph = 0, gch = 0;   // gch: the chunk's first atom, numbered in the CTA
        bool ab = false;
        // class words (not PRE) of this thread in atom t: row c0, its words
        // [2 * part, 2 * part + 2) with MT = 2 (2 R items), rows c0 and
        // c0 + 128 whole with MT = 1
        const int c0 = MT == 2 ? urow % p.R : urow, part = MT == 2 ? urow / p.R : 0;
        auto class_words = [&](int c, int t) {   // ordinary loads: an earlier kernel may write cls until grid_wait
            const bool ok = part < 2 && c < p.C && t * 4 < p.W;
            const uint32_t *w = p.cls + (int64_t)(ok ? c : 0) * p.W + (ok ? t * 4 : 0);
            if (!ok) return make_uint4(0, 0, 0, 0);
            if (MT == 1) return __ldcg(reinterpret_cast<const uint4 *>(w));
            const uint2 h = __ldcg(reinterpret_cast<const uint2 *>(w + part * 2));
            return make_uint4(h.x, h.y, 0, 0);
        };
        const int tu0 = ch0 * 2 * HP_CHUNK, tun = min(ch1 * 2 * HP_CHUNK, 2 * p.nt) - tu0;   // a unit's atoms
        uint4 cn0, cn1;   // class words of this warp's next atom
        if (!PRE) {
            cn0 = class_words(c0, tu0 + (int)grp % tun);
            if (MT == 1) cn1 = class_words(c0 + 128, tu0 + (int)grp % tun);
        }
        for (int64_t u = u0; u < units && !ab; u += ustep) {
            for (int ch = ch0; ch < ch1 && !ab; ch++) {
                const bool okq = mbar_wait(qfull(qs), qph, abort_flag);
                if (!__all_sync(0xffffffffu, okq)) { ab = true; break; }
                const uint8_t *qrow = sQ + qs * QCH + urow * 128;
                const int na = chunk_atoms(ch);
                const int a0 = (int)((grp - gch) % (uint32_t)AS);
                if (a0 >= na && lane == 0) mbar_arrive(qempty(qs));
                for (int a = a0; a < na; a += AS) {
                    const int t = ch * 2 * HP_CHUNK + a;
                    const uint32_t g = gch + (uint32_t)a;
                    const uint4 qw = *reinterpret_cast<const uint4 *>(qrow + ((a ^ (urow & 7)) << 4));
                    const uint32_t ws[4] = {qw.x, qw.y, qw.z, qw.w};
                    uint32_t b[32];
#pragma unroll
                    for (int i = 0; i < 4; i++)
#pragma unroll
                        for (int j = 0; j < 8; j++) b[8 * i + j] = hp_signs(ws[i], j);
                    const uint4 cw0 = cn0, cw1 = cn1;
                    if (!PRE) {   // AS atoms on, in this unit or a following one
                        const int tn = tu0 + (t - tu0 + AS) % tun;
                        cn0 = class_words(c0, tn);
                        if (MT == 1) cn1 = class_words(c0 + 128, tn);
                    }
                    const int buf = g % NAB;
                    const bool oke = mbar_wait_fast(aempty(buf), ((g / NAB) & 1) ^ 1, abort_flag);   // its last MMAs
                    if (!__all_sync(0xffffffffu, oke)) { ab = true; break; }
                    tc_fence_after();
                    __syncwarp();   // converged for the warp-wide store
                    hp_tmem_st32(tcol + (uint32_t)(buf * MT * 32), b);
                    if (!PRE) {
                        const uint4 m = t * 4 < p.W ? *reinterpret_cast<const uint4 *>(smask + t * 4) : make_uint4(0, 0, 0, 0);
                        uint8_t *at = sB + buf * atom_bytes;
                        if (MT == 2) {
                            if (part < 2) hp_expand_row<2>(at, c0, part * 4, cw0, part ? make_uint4(m.z, m.w, 0, 0) : m);
                        } else {
                            if (c0 < p.R) hp_expand_row<4>(at, c0, 0, cw0, m);
                            if (c0 + 128 < p.R) hp_expand_row<4>(at, c0 + 128, 0, cw1, m);
                        }
                        fence_async_smem();
                    }
                    h_tmem_st_wait();   // the query columns landed before the MMAs read them
                    tc_fence_before();
                    __syncwarp();
                    // the chunk's slot is given back only here, past the store
                    // that consumed its last words: ahead of the wait for the
                    // buffer the loads could still be outstanding
                    if (lane == 0) {
                        mbar_arrive(afull(buf));
                        if (a + AS >= na) mbar_arrive(qempty(qs));
                    }
                }
                gch += (uint32_t)na;
                if (++qs == HP_QB) { qs = 0; qph ^= 1; }
            }
        }
    } else if (warp - HP_EPI0 < 4 * MT) {  // -------------- epilogue warps 16 .. 15 + 4 * MT
        const int e = warp - HP_EPI0;
        const uint32_t tlane = (uint32_t)((warp & 3) * 32) << 16;
        int d2 = 0;
        uint32_t d2ph = 0;
        for (int64_t u = u0; u < units; u += ustep) {
            const bool okd = mbar_wait(d2full(d2), d2ph, abort_flag);
            if (!__all_sync(0xffffffffu, okd)) break;
            tc_fence_after();
            const uint32_t dcol = tmem + tlane + (uint32_t)((d2 * MT + (e >> 2)) * RS);
            if (S == 1 && !HAM) {
                finish_scores(u * UROWS + e * 32,
                              [&](int col, uint32_t(&v)[8]) { hp_tmem_ld8(dcol + (uint32_t)col, v); });
            } else if (S == 1) {
                finish(u * UROWS + e * 32, s_out + e * (HP_OUT / 4), [&](int j, uint32_t(&v)[32]) { tmem_ld32(dcol + (uint32_t)(j * 32), v); });
            } else {   // this rank's partial sums, [column][row of the unit], over the rings (all consumed)
                float *dump = reinterpret_cast<float *>(smem) + e * 32 + lane;
                for (int j = 0; j * 32 < p.R; j++) {
                    uint32_t v[32];
                    tmem_ld32(dcol + (uint32_t)(j * 32), v);
#pragma unroll
                    for (int i = 0; i < 32; i++)
                        if (j * 32 + i < p.R) dump[(j * 32 + i) * UROWS] = __uint_as_float(v[i]);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(d2empty(d2));
            if (++d2 == ND2) { d2 = 0; d2ph ^= 1; }
        }
    }

    __syncwarp();
    if (S > 1) {   // one unit per cluster: every rank's sums are in its shared memory
        hp_cluster_sync();
        const int e = warp - HP_EPI0;
        if (e >= 0 && e < 4 * MT && e % S == rank && u0 < units) {
            const uint32_t base = su32(smem) + (uint32_t)(e * 32 + lane) * 4u;
            // the ranks' sums of this row, sixteen columns at a time, into this
            // rank's own copy (no other rank reads these rows)
            float *own = reinterpret_cast<float *>(smem) + e * 32 + lane;
            for (int col = 0; col < p.R; col += 16) {   // R is a multiple of 16
                float t[16];
#pragma unroll
                for (int i = 0; i < 16; i++) t[i] = 0.f;
                for (int k = 0; k < S; k++)
#pragma unroll
                    for (int i = 0; i < 16; i++)
                        t[i] += hp_ld_cluster(base + (uint32_t)((col + i) * UROWS) * 4u, (uint32_t)k);
#pragma unroll
                for (int i = 0; i < 16; i++) own[(col + i) * UROWS] = t[i];
            }
            auto sums = [&](int col, uint32_t *v, auto count) {
#pragma unroll
                for (int i = 0; i < decltype(count)::value; i++)
                    v[i] = col + i < p.R ? __float_as_uint(own[(col + i) * UROWS]) : 0u;
            };
            if (HAM)
                finish(u0 * UROWS + e * 32, s_out + e * (HP_OUT / 4),
                       [&](int j, uint32_t(&v)[32]) { sums(j * 32, v, HpInt<32>()); });
            else
                finish_scores(u0 * UROWS + e * 32, [&](int col, uint32_t(&v)[8]) { sums(col, v, HpInt<8>()); });
        }
        __syncwarp();
        hp_cluster_sync();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

}  // namespace tc
}  // namespace hdc
