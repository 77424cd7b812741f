// Level-ID encoding (Sec. 4.2 Algorithmic Choice: ID-based encoding as the
// alternative to random projection; Sec. 5.3: Micro-HD-Classification's
// Level-ID encoder and its N_LEVELS knob).
//
//   level(x_f) = clamp(floor((x_f - lo) * scale), 0, L-1)     FP32, as written
//   s_d        = sum_f ID_f[d] * LEVEL_{level(x_f)}[d]          (+-1 elements)
//   bit_d      = s_d < 0                                        (sign(0) = +1)
// With bit 1 = element -1, the product of two elements is -1 exactly when
// their bits differ, so s_d = F - 2 cnt_d with cnt_d = #{f : id_f,d != lv_f,d}
// and bit_d = cnt_d > floor(F/2): a per-dimension majority of XORs.
//
// Level hypervectors: level l has the bit of `hi_hv` at dim d when
// l >= flip[d], else the bit of `lo_hv` (flip[d] in 1..L-1: level 0 is lo_hv,
// level L-1 is hi_hv, neighbouring levels differ in the dims that switch
// between them).  ID and level rows are compacted to the kept dims at
// model preparation, like the base rows of the random projection.
//
// Encode kernel of medium batches: one block per (32 queries, 32 words); the block stages its
// word slice of every ID row and every level row in shared memory.  A warp
// takes four queries at a time (four independent counter chains, each ID
// word loaded once for the four), a lane one word (32 dims): lane j
// quantises feature f0 + j of each query, the warp broadcasts the levels by
// shuffle, and each lane adds id ^ level rows into a bit-sliced counter per
// query (carry-save adders over groups of 16 rows with the planes of weight
// 1, 2, 4 and 8 as carry-save state, then a ripple-carry add of the
// weight-16 row into planes sized for F), then compares the counter against
// floor(F/2) bit-sliced.  The next 32 features of each query are loaded
// while the current ones are counted.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "bitslice.cuh"
#include "hdc_internal.cuh"

namespace hdc {
namespace {

constexpr int LQ = 32;       // queries per block
constexpr int LWC = 32;      // words per block (one per lane)
constexpr int LWARPS = 8;
// counter planes of weight 16, 32, ...: HP of them hold floor(F / 16) < 2^HP
__host__ __device__ constexpr int hp_for(int F) { return F < 1024 ? 6 : 9; }

__device__ __forceinline__ int quant_level(float x, float lo, float scale, int L)
{
    // separate FP32 rounding of the difference and the product (no FMA), as the oracle
    const float t = __fmul_rn(__fsub_rn(x, lo), scale);
    if (t >= (float)L) return L - 1;
    if (t > 0.f) return (int)t;  // floor of a positive value
    return 0;                    // t <= 0, or NaN
}

// The counter of one query and lane: planes c1, c2, c4, c8 (weights 1, 2,
// 4, 8) and hp[k] (weight 16 * 2^k); bit position i of the planes spells
// the count of dim i in binary.
template <int HP>
struct Counter {
    uint32_t c1, c2, c4, c8, hp[HP];
};

// Add 16 rows of weight 1: a carry-save tree (15 full adders) to one row of
// weight 16, then a ripple-carry add of it into hp.
template <int HP>
__device__ __forceinline__ void add16(Counter<HP> &k, const uint32_t (&r)[16])
{
    uint32_t c = csa16(k.c1, k.c2, k.c4, k.c8, r);
#pragma unroll
    for (int i = 0; i < HP; i++) {
        const uint32_t t = k.hp[i] & c;
        k.hp[i] ^= c;
        c = t;
    }
}

// Add one row of weight 1 (ripple carry through every plane).
template <int HP>
__device__ __forceinline__ void add1(Counter<HP> &k, uint32_t c)
{
    uint32_t t = k.c1 & c; k.c1 ^= c; c = t;
    t = k.c2 & c; k.c2 ^= c; c = t;
    t = k.c4 & c; k.c4 ^= c; c = t;
    t = k.c8 & c; k.c8 ^= c; c = t;
#pragma unroll
    for (int i = 0; i < HP; i++) {
        const uint32_t u = k.hp[i] & c;
        k.hp[i] ^= c;
        c = u;
    }
}

// count > T per bit position, from the most significant plane down.
template <int HP>
__device__ __forceinline__ uint32_t greater(const Counter<HP> &k, uint32_t T)
{
    uint32_t gt = 0, eq = 0xffffffffu;
#pragma unroll
    for (int i = HP - 1; i >= 0; i--) {
        const uint32_t cp = k.hp[i];
        if ((T >> (i + 4)) & 1u) eq &= cp;
        else { gt |= eq & cp; eq &= ~cp; }
    }
    const uint32_t pl[4] = {k.c8, k.c4, k.c2, k.c1};
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const uint32_t cp = pl[i];
        if ((T >> (3 - i)) & 1u) eq &= cp;
        else { gt |= eq & cp; eq &= ~cp; }
    }
    return gt;
}

// Most varying dims of a 1,024-dim slice that levelid_count_kernel takes.  Random
// level end points differ in 512 +- 16; the rows' kernel takes the same time for
// any number, so where nearly all vary it is the faster one again with few
// features (39,000 queries, 1,024 varying dims: 784 features, 128 levels 528 / 651
// us; 660, 16 levels 431 / 358).
__host__ __device__ constexpr int most_varying(int F) { return F >= 740 ? 1024 : 600; }

// Whether levelid_count_kernel leaves a slice out: too many dims vary, or one
// differs more than once over the levels (a level table of the caller's own).
// For one warp, lane j on word j; calls at(dims, l) with the dims of word j that
// differ between levels l - 1 and l.
template <typename At>
__device__ __forceinline__ bool left_out(const uint32_t *slv, int F, int L, int j, At &&at)
{
    uint32_t seen = 0, twice = 0, prev = slv[j];
    for (int l = 1; l < L; l++) {
        const uint32_t cur = slv[l * LWC + j], ch = cur ^ prev;
        if (ch) at(ch, l);
        twice |= ch & seen;
        seen |= ch;
        prev = cur;
    }
    __syncwarp();
    return __any_sync(0xffffffffu, twice != 0) || __reduce_add_sync(0xffffffffu, __popc(seen)) > most_varying(F);
}

// A warp encodes QW queries at once (independent counter chains; each ID
// word loaded once for all of them).
constexpr int QW = 4;
// per warp: the level-row offsets (level x LWC words) of its QW queries'
// current 32 features, read back 16 at a time as broadcasts
constexpr size_t LOFF_BYTES = (size_t)LWARPS * QW * 32 * 4;

// REST: only the word slices that levelid_count_kernel leaves out, with a grid
// that may be shorter than the queries.
template <int HP, bool REST>
__global__ void __launch_bounds__(LWARPS * 32) levelid_encode_kernel(const float *__restrict__ X, int64_t N, int F,
                                                                   int L, int W, float lo, float scale,
                                                                   const uint32_t *__restrict__ id,
                                                                   const uint32_t *__restrict__ lv,
                                                                   uint32_t *__restrict__ H)
{
    extern __shared__ uint32_t lsm[];
    uint32_t *sid = lsm;                          // F x LWC
    uint32_t *slv = lsm + (size_t)F * LWC;        // L x LWC
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int *soff = reinterpret_cast<int *>(lsm + (size_t)(F + L) * LWC) + warp * (QW * 32);   // [QW][32]
    const int w0 = blockIdx.y * LWC;
    const int nw = min(LWC, W - w0);
    auto stage_levels = [&]() {
        for (int i = threadIdx.x; i < L * LWC; i += blockDim.x) {
            const int l = i / LWC, j = i % LWC;
            slv[i] = j < nw ? lv[(int64_t)l * W + w0 + j] : 0u;
        }
    };
    if (REST) {
        stage_levels();
        __syncthreads();
        bool left = false;
        if (warp == 0) left = left_out(slv, F, L, lane, [](uint32_t, int) {});
        if (!__syncthreads_or(left)) return;
    }
    for (int i = threadIdx.x; i < F * LWC; i += blockDim.x) {
        const int f = i / LWC, j = i % LWC;
        sid[i] = j < nw ? id[(int64_t)f * W + w0 + j] : 0u;
    }
    if (!REST) stage_levels();
    __syncthreads();
    const uint32_t T = (uint32_t)F >> 1;
    int64_t tile = blockIdx.x;
    do {
        for (int qb = warp * QW; qb < LQ; qb += LWARPS * QW) {
            const int64_t q0 = tile * LQ + qb;
            if (q0 >= N) break;                       // warp-uniform
            Counter<HP> cnt[QW];
    #pragma unroll
            for (int a = 0; a < QW; a++) {
                cnt[a].c1 = cnt[a].c2 = cnt[a].c4 = cnt[a].c8 = 0;
    #pragma unroll
                for (int k = 0; k < HP; k++) cnt[a].hp[k] = 0;
            }
            // feature f0 + lane of each query, loaded one 32-feature batch ahead
            // so the quantisation does not wait on device memory
            float xn[QW];
    #pragma unroll
            for (int a = 0; a < QW; a++) xn[a] = (lane < F && q0 + a < N) ? X[(q0 + a) * (int64_t)F + lane] : 0.f;
            for (int f0 = 0; f0 < F; f0 += 32) {
                const int f = f0 + lane;
                // level-row offset of feature f of each query (rows past N: level 0, not stored)
    #pragma unroll
                for (int a = 0; a < QW; a++) {
                    soff[a * 32 + lane] = (f < F && q0 + a < N) ? quant_level(xn[a], lo, scale, L) * LWC : 0;
                    const int fn = f + 32;
                    xn[a] = (fn < F && q0 + a < N) ? X[(q0 + a) * (int64_t)F + fn] : 0.f;
                }
                __syncwarp();
                const int nf = min(32, F - f0);
                int j = 0;
                for (; j + 16 <= nf; j += 16) {
                    uint32_t idw[16];
    #pragma unroll
                    for (int u = 0; u < 16; u++) idw[u] = sid[(f0 + j + u) * LWC + lane];
    #pragma unroll
                    for (int a = 0; a < QW; a++) {
                        int o[16];   // four 16-byte broadcasts (j is a multiple of 16)
                        const int4 *o4 = reinterpret_cast<const int4 *>(soff + a * 32 + j);
    #pragma unroll
                        for (int v = 0; v < 4; v++) {
                            const int4 t = o4[v];
                            o[4 * v] = t.x; o[4 * v + 1] = t.y; o[4 * v + 2] = t.z; o[4 * v + 3] = t.w;
                        }
                        uint32_t r[16];
    #pragma unroll
                        for (int u = 0; u < 16; u++) r[u] = idw[u] ^ slv[o[u] + lane];
                        add16(cnt[a], r);
                    }
                }
                for (; j < nf; j++) {
                    const uint32_t idw = sid[(f0 + j) * LWC + lane];
    #pragma unroll
                    for (int a = 0; a < QW; a++) add1(cnt[a], idw ^ slv[soff[a * 32 + j] + lane]);
                }
                __syncwarp();   // the batch's offsets are read before the next batch writes them
            }
    #pragma unroll
            for (int a = 0; a < QW; a++)
                if (q0 + a < N && lane < nw)
                    H[(q0 + a) * (int64_t)W + w0 + lane] = greater(cnt[a], T);
        }
        tile += gridDim.x;
    } while (REST && tile * LQ < N);
}

// ---- few queries ------------------------------------------------------------
//
// One wave of the kernel above is latency: the rows staged a load at a time, then
// 32 features after another whose values come from device memory, in one warp
// where there are four queries.  Here the rows are staged by asynchronous
// copies while all of the queries' levels are formed, and a warp takes Q1
// queries: one while the blocks fit the SMs, four then.  One query, 561 x 4,928,
// 128 levels 48 -> 11 us; 1,000, 617 x 1,024 62 -> 15 (four a warp, 3,000: 64 -> 41).
template <int HP, int Q1>
__global__ void __launch_bounds__(LWARPS * 32) levelid_few_kernel(const float *__restrict__ X, int64_t N, int F, int L, int W,
                                                                float lo, float scale, const uint32_t *__restrict__ id,
                                                                const uint32_t *__restrict__ lv, uint32_t *__restrict__ H)
{
    extern __shared__ __align__(16) uint32_t lsm[];
    const uint32_t *sid = lsm, *slv = lsm + (size_t)F * LWC;         // F x LWC, L x LWC
    const int Fp = (F + 3) / 4 * 4;
    int *soff = reinterpret_cast<int *>(lsm + (size_t)(F + L) * LWC);   // [LWARPS * Q1][Fp] level-row offsets
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int w0 = blockIdx.y * LWC, nw = min(LWC, W - w0);          // W is a multiple of 4
    for (int i = threadIdx.x; i < (F + L) * (LWC / 4); i += LWARPS * 32) {
        const int r = i / (LWC / 4), c = i % (LWC / 4) * 4;
        const uint32_t *src = (r < F ? id + (int64_t)r * W : lv + (int64_t)(r - F) * W) + w0 + c;
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(lsm + r * LWC + c);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(c < nw ? src : id), "r"(c < nw ? 16 : 0));
    }
    asm volatile("cp.async.commit_group;");
    const int64_t q0 = ((int64_t)blockIdx.x * LWARPS + warp) * Q1;   // this warp's queries
    int *off = soff + warp * Q1 * Fp;
    // a step's loads all in flight, the partial one's too: left to the loop's
    // remainder they waited for memory up to three times more a query, so that
    // F = 225 .. 255 took longer than the kernel above (3,000 x 232 x 500: 28.1 us,
    // 23.9 there; 17.0 so)
    constexpr int FU = Q1 == 1 ? 8 : 4;
    for (int f0 = lane; f0 < F; f0 += 32 * FU) {
        float x[Q1][FU];
#pragma unroll
        for (int a = 0; a < Q1; a++)
#pragma unroll
            for (int u = 0; u < FU; u++)
                x[a][u] = f0 + 32 * u < F && q0 + a < N ? __ldg(X + (q0 + a) * F + f0 + 32 * u) : 0.f;
#pragma unroll
        for (int a = 0; a < Q1; a++)
#pragma unroll
            for (int u = 0; u < FU; u++)   // rows past N: not stored
                if (f0 + 32 * u < F) off[a * Fp + f0 + 32 * u] = quant_level(x[a][u], lo, scale, L) * LWC;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    if (q0 >= N) return;
    Counter<HP> cnt[Q1];
#pragma unroll
    for (int a = 0; a < Q1; a++) {
        cnt[a].c1 = cnt[a].c2 = cnt[a].c4 = cnt[a].c8 = 0;
#pragma unroll
        for (int k = 0; k < HP; k++) cnt[a].hp[k] = 0;
    }
    int f = 0;
    for (; f + 16 <= F; f += 16) {
        uint32_t idw[16];
#pragma unroll
        for (int u = 0; u < 16; u++) idw[u] = sid[(f + u) * LWC + lane];
#pragma unroll
        for (int a = 0; a < Q1; a++) {
            const int4 *o4 = reinterpret_cast<const int4 *>(off + a * Fp + f);
            uint32_t r[16];
#pragma unroll
            for (int v = 0; v < 4; v++) {
                const int4 t = o4[v];
                r[4 * v] = idw[4 * v] ^ slv[t.x + lane];
                r[4 * v + 1] = idw[4 * v + 1] ^ slv[t.y + lane];
                r[4 * v + 2] = idw[4 * v + 2] ^ slv[t.z + lane];
                r[4 * v + 3] = idw[4 * v + 3] ^ slv[t.w + lane];
            }
            add16(cnt[a], r);
        }
    }
    for (; f < F; f++)
#pragma unroll
        for (int a = 0; a < Q1; a++) add1(cnt[a], sid[f * LWC + lane] ^ slv[off[a * Fp + f] + lane]);
#pragma unroll
    for (int a = 0; a < Q1; a++)
        if (q0 + a < N && lane < nw) H[(q0 + a) * (int64_t)W + w0 + lane] = greater(cnt[a], (uint32_t)F >> 1);
}

// ---- many queries ----------------------------------------------------------
//
// The kernel above adds F rows into W words whatever the levels are.  Half of
// the random dims need no work per query: where the level end points agree the
// bit is a constant of the model.  For the others, with x_f = id_f ^ lo and the
// dim's switch level t, cnt = popc over the features of x ^ [l_f >= t]: F / 32
// words a dim instead of F rows a word.  A thread holds one query: its levels as
// bit planes over the features (7 planes of F / 32 words, in registers); per
// level t one majority operation a plane and word gives [l_f >= t]; per dim that
// switches there, carry-save adders and popcounts.  The dims' words are the same
// for every thread (broadcast reads of shared memory), sorted by t.  Per (query,
// varying dim) 40 logic operations and 10 POPC at 20 words, where the rows above
// take 4.7 F / 32 = 91 operations for every dim.
// 262,144 x 617 x 1,024: 128 levels 2,062 -> 1,080 us, 16 levels 1,998 -> 831;
// 60,000 x 617 x 10,000, 128 levels 4,707 -> 2,514.  Bound by the logic pipe (69 %
// of its slots; two warps a scheduler, 240 registers a thread).

constexpr int CT = 256;                 // threads of a block
constexpr int CPL = 7;                  // level planes: L <= 128
constexpr int CD = LWC * 32;            // dims of a block's slice

// 32-feature words a scratch group holds (NFW a multiple), shared words from dim
// to dim, scratch rows (a group's planes; 32 result words and a row of zeros).
template <int NFW> __host__ __device__ constexpr int c_group() { return NFW % 5 == 0 ? 5 : 4; }
template <int NFW> __host__ __device__ constexpr int c_pitch() { return (NFW + 3) / 4 * 4; }
template <int NFW> __host__ __device__ constexpr int c_rows()
{
    return CPL * c_group<NFW>() > 33 ? CPL * c_group<NFW>() : 33;
}
template <int NFW>
constexpr size_t count_smem()
{
    return (size_t)CD * c_pitch<NFW>() * 4 + (size_t)c_rows<NFW>() * CT * 4 + CD * 2 + LWC * 8 + (128 + 1) * 4 + 128 * 4;
}

// Bit i of lane j's result: bit j of lane i's word (blocks off the diagonal
// exchanged, halving).
__device__ __forceinline__ uint32_t transpose32(uint32_t x, int lane)
{
#pragma unroll
    for (int k = 4; k >= 0; k--) {
        const int s = 1 << k;
        const uint32_t m = 0xffffffffu / ((1u << s) + 1u);
        const uint32_t y = __shfl_xor_sync(0xffffffffu, x, s);
        x = lane & s ? (x & ~m) | ((y >> s) & m) : (x & m) | ((y & m) << s);
    }
    return x;
}

// One round of full adders over the N words of v: a sum of weight 1 for every
// three, then the words left over; the carries in c.
template <int N>
__device__ __forceinline__ void adders(const uint32_t (&v)[N], uint32_t (&sum)[N / 3 + N % 3], uint32_t (&c)[N / 3])
{
#pragma unroll
    for (int i = 0; i < N / 3; i++) csa(c[i], sum[i], v[3 * i], v[3 * i + 1], v[3 * i + 2]);
#pragma unroll
    for (int i = 0; i < N % 3; i++) sum[N / 3 + i] = v[N - N % 3 + i];
}

template <int N>
__device__ __forceinline__ int pops(const uint32_t (&v)[N])
{
    int n = 0;
#pragma unroll
    for (int i = 0; i < N; i++) n += __popc(v[i]);
    return n;
}

// Set bits of v: two rounds of adders on the words, one on the carries, popcounts
// of what is left.  Adders run on the logic pipe (16 lanes a clock, two
// operations each), popcounts on another at a quarter of its rate: 20 words are
// 40 operations with the differences and 10 popcounts, 80 clocks of either;
// reduced as far as it goes (14 adders, 6 popcounts) 1,099 us against 1,080.
template <int N>
__device__ __forceinline__ int weigh(const uint32_t (&v)[N])
{
    constexpr int S = N / 3 + N % 3, C = N / 3, S2 = S / 3 + S % 3, C2 = S / 3, T = C + C2;
    static_assert(N >= 8, "three carries at least");
    uint32_t sum[S], c[C], sum2[S2], c2[C2], twos[T], two[T / 3 + T % 3], four[T / 3];
    adders<N>(v, sum, c);
    adders<S>(sum, sum2, c2);
#pragma unroll
    for (int i = 0; i < T; i++) twos[i] = i < C ? c[i] : c2[i < C ? 0 : i - C];
    adders<T>(twos, two, four);
    return pops(sum2) + 2 * pops(two) + 4 * pops(four);
}

// Set bits of a[i] ^ b[i].
template <int NFW>
__device__ __forceinline__ int count_bits(const uint32_t (&a)[NFW], const uint32_t *b)
{
    uint32_t y[c_pitch<NFW>()], x[NFW];
#pragma unroll
    for (int i = 0; i < c_pitch<NFW>() / 4; i++) {
        const uint4 v = reinterpret_cast<const uint4 *>(b)[i];
        y[4 * i] = v.x;
        y[4 * i + 1] = v.y;
        y[4 * i + 2] = v.z;
        y[4 * i + 3] = v.w;
    }
#pragma unroll
    for (int i = 0; i < NFW; i++) x[i] = a[i] ^ y[i];
    return weigh<NFW>(x);
}

// Block (x, y): word slice y; the warps of all blocks of a slice take 32 queries
// each in turn.  Slices that left_out() names stay for the kernel above.
template <int NFW>
__global__ void __launch_bounds__(CT, NFW <= 8 ? 2 : 1) levelid_count_kernel(const float *__restrict__ X, int64_t N, int F,
                                                                             int L, int W, float lo, float scale,
                                                                             const uint32_t *__restrict__ id,
                                                                             const uint32_t *__restrict__ lv,
                                                                             uint32_t *__restrict__ H)
{
    constexpr int P = c_pitch<NFW>(), GF = c_group<NFW>(), ROWS = c_rows<NFW>();
    extern __shared__ __align__(16) uint32_t csm[];
    uint32_t *sb = csm;                                              // [CD][P]: x_f of the varying dims
    uint32_t *scr = sb + CD * P;                                     // [ROWS][CT]: planes, then result words
    // [CD] place of a dim (0xffff: constant); then the byte offset of its result
    // word in a thread's column (a multiple of CT * 4) + its bit, 32 rows on when constant
    uint16_t *spos = reinterpret_cast<uint16_t *>(scr + ROWS * CT);
    uint32_t *slo = reinterpret_cast<uint32_t *>(spos + CD), *sconst = slo + LWC;   // level 0; bits of the constant dims
    int32_t *first = reinterpret_cast<int32_t *>(sconst + LWC);      // [129] first dim of a level
    int32_t *cur = first + 129;                                      // [128]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int w0 = blockIdx.y * LWC, nw = min(LWC, W - w0);
    uint32_t *slv = scr;   // [L][LWC], for the set-up
    for (int i = tid; i < L * LWC; i += CT) slv[i] = i % LWC < nw ? lv[(int64_t)(i / LWC) * W + w0 + i % LWC] : 0u;
    for (int i = tid; i < CD; i += CT) spos[i] = 0xffff;
    if (tid < 128) cur[tid] = 0;
    __syncthreads();
    bool odd = false;
    if (warp == 0) {
        slo[lane] = slv[lane];
        odd = left_out(slv, F, L, lane, [&](uint32_t ch, int l) {
            for (atomicAdd(&cur[l], __popc(ch)); ch; ch &= ch - 1) spos[lane * 32 + __ffs(ch) - 1] = (uint16_t)l;
        });
    }
    if (__syncthreads_or(odd)) return;
    if (warp == 0) {   // levels 4 lane .. 4 lane + 3
        int n[4], sum = 0;
#pragma unroll
        for (int i = 0; i < 4; i++) n[i] = cur[4 * lane + i], sum += n[i];
        int at = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, at, o);
            if (lane >= o) at += y;
        }
        if (lane == 31) first[128] = at;
        at -= sum;
#pragma unroll
        for (int i = 0; i < 4; i++) {
            first[4 * lane + i] = cur[4 * lane + i] = at;
            at += n[i];
        }
    }
    __syncthreads();
    for (int d = tid; d < CD; d += CT)
        if (spos[d] != 0xffff) spos[d] = (uint16_t)atomicAdd(&cur[spos[d]], 1);
    __syncthreads();
    for (int w = warp; w < LWC; w += CT / 32) {
        const int pos = spos[w * 32 + lane];
        int n = 0;
        for (int fw = 0; fw < NFW; fw++) {
            const int f = fw * 32 + lane;
            const uint32_t x = transpose32(f < F && w < nw ? id[(int64_t)f * W + w0 + w] ^ slo[w] : 0u, lane);
            if (pos != 0xffff) sb[pos * P + fw] = x;
            else n += __popc(x);
        }
        const uint32_t bits = __ballot_sync(0xffffffffu, pos == 0xffff && n > F / 2);
        if (lane == 0) sconst[w] = bits;
        static_assert(CT * 4 >= 32 && 32 * CT * 4 + 31 < 65536, "a dim's place in 16 bits");
        spos[w * 32 + lane] = (uint16_t)(pos == 0xffff ? 32 * CT * 4 : (pos >> 5) * (CT * 4) + (pos & 31));
    }
    __syncthreads();

    const float top = (float)(L - 1);
    const int half = F >> 1;
    const bool wide = ((uintptr_t)H & 15) == 0;
    uint32_t *mine = scr + tid;
    for (int64_t q0 = ((int64_t)warp * gridDim.x + blockIdx.x) * 32; q0 < N; q0 += (int64_t)gridDim.x * CT) {
        // the levels' planes: lane j quantises feature j of a 32-feature word for
        // all 32 queries (byte b of p[k]: query 8 b + k), the transposition hands
        // each query its word
        uint32_t pl[CPL][NFW];
#pragma unroll
        for (int g = 0; g < NFW / GF; g++) {
#pragma unroll 1
            for (int ff = 0; ff < GF; ff++) {
                const int f = (g * GF + ff) * 32 + lane;
                const float *src = X + q0 * F + f;
                const int nq = f < F ? (int)min((int64_t)32, N - q0) : 0;
                if (q0 + lane < N && f - lane + 64 < F)   // the row of lane's query, two words on
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(X + (q0 + lane) * F + f - lane + 64));
                float v[32];
#pragma unroll
                for (int i = 0; i < 32; i++) v[i] = i < nq ? __ldg(src + i * F) : lo;
                uint32_t p[8];
#pragma unroll
                for (int k = 0; k < 8; k++) {
                    p[k] = 0;
#pragma unroll
                    for (int b = 0; b < 4; b++) {
                        const float x = __fmul_rn(__fsub_rn(v[8 * b + k], lo), scale);   // as quant_level
                        p[k] |= __float2uint_rz(fminf(fmaxf(x, 0.f), top)) << (8 * b);
                    }
                }
#pragma unroll
                for (int b = 0; b < CPL; b++) {
                    uint32_t word = 0;
#pragma unroll
                    for (int k = 0; k < 8; k++)
                        word |= (k >= b ? p[k] << (k - b) : p[k] >> (b - k)) & (0x01010101u << k);
                    mine[(ff * CPL + b) * CT] = transpose32(word, lane);
                }
            }
#pragma unroll
            for (int ff = 0; ff < GF; ff++)
#pragma unroll
                for (int b = 0; b < CPL; b++) pl[b][g * GF + ff] = mine[(ff * CPL + b) * CT];
        }
        // result bits in the dims' sorted order, the first of 32 on top
        uint32_t res = 0;
        int d = 0;
        for (int t = 1; t < L; t++) {
            const int end = first[t + 1];
            if (d == end) continue;
            uint32_t a[NFW];   // l_f >= t: from the lowest plane up, and / or by the bit of t
#pragma unroll
            for (int b = 0; b < CPL; b++) {
                const uint32_t m = (uint32_t)(t >> b & 1) - 1u;
#pragma unroll
                for (int i = 0; i < NFW; i++) a[i] = b == 0 ? pl[0][i] | m : (a[i] & pl[b][i]) | (m & (a[i] | pl[b][i]));
            }
            auto put = [&](int s, int at) {   // s < 0: the bit of dim `at` is set
                res = __funnelshift_l((uint32_t)s, res, 1);
                if ((at & 31) == 31) mine[(at >> 5) * CT] = res;
            };
            if constexpr (NFW <= 20) {   // two dims at once: their chains are independent
                for (; d + 2 <= end; d += 2) {
                    const int s0 = half - count_bits<NFW>(a, sb + d * P), s1 = half - count_bits<NFW>(a, sb + (d + 1) * P);
                    put(s0, d);
                    put(s1, d + 1);
                }
            }
            for (; d < end; d++) put(half - count_bits<NFW>(a, sb + d * P), d);
        }
        if (d & 31) mine[(d >> 5) * CT] = res << (32 - (d & 31));
        mine[32 * CT] = 0;
        // back to the dims' own order
        if (q0 + lane < N) {
            uint32_t *out = H + (q0 + lane) * W + w0;
            for (int w4 = 0; w4 < nw; w4 += 4) {   // W is a multiple of 4
                uint32_t o[4];
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    const uint4 *e = reinterpret_cast<const uint4 *>(spos + (w4 + k) * 32);
                    uint32_t word = 0;
#pragma unroll
                    for (int j = 3; j >= 0; j--) {
                        const uint4 e8 = e[j];
                        const uint32_t e2[4] = {e8.x, e8.y, e8.z, e8.w};
#pragma unroll
                        for (int i = 7; i >= 0; i--) {
                            const uint32_t at = i & 1 ? e2[i / 2] >> 16 : e2[i / 2];
                            const uint32_t r = *reinterpret_cast<const uint32_t *>(
                                reinterpret_cast<const uint8_t *>(mine) + (at & (0xffffu & ~(CT * 4u - 1))));
                            word = __funnelshift_l(__funnelshift_l(0u, r, at), word, 1);
                        }
                    }
                    o[k] = word | sconst[w4 + k];
                }
                if (wide) {
                    *reinterpret_cast<uint4 *>(out + w4) = make_uint4(o[0], o[1], o[2], o[3]);
                } else {
#pragma unroll
                    for (int k = 0; k < 4; k++) out[w4 + k] = o[k];
                }
            }
        }
    }
}

// Model preparation: one thread per output word of the compacted rows,
// packing the caller's unpacked bytes (nonzero = the element -1) of the
// kept dims d = s0 + k*stride.
//   rows [0, F):      ID row f (id_bits: F x D bytes)
//   rows [F, F + L):  level l, bit d = l >= flip[d] ? hi[d] : lo[d]
__global__ void levelid_prepare_kernel(const uint8_t *__restrict__ id_bits, const uint8_t *__restrict__ lo_bits,
                                       const uint8_t *__restrict__ hi_bits, const int32_t *__restrict__ flip, int F,
                                       int L, int64_t D, int64_t s0, int64_t stride, int64_t Dk, int Wk,
                                       uint32_t *__restrict__ id, uint32_t *__restrict__ lv)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)(F + L) * Wk) return;
    const int r = (int)(i / Wk), kw = (int)(i % Wk);
    uint32_t word = 0;
    for (int j = 0; j < 32; j++) {
        const int64_t k = (int64_t)kw * 32 + j;
        if (k >= Dk) break;
        const int64_t d = s0 + k * stride;
        uint8_t b;
        if (r < F) {
            b = id_bits[(int64_t)r * D + d];
        } else {
            const int l = r - F;
            b = l >= flip[d] ? hi_bits[d] : lo_bits[d];
        }
        word |= (uint32_t)(b != 0) << j;
    }
    if (r < F) id[(int64_t)r * Wk + kw] = word;
    else lv[(int64_t)(r - F) * Wk + kw] = word;
}

__global__ void flip_check_kernel(const int32_t *__restrict__ flip, int D, int L, int *__restrict__ bad)
{
    for (int d = blockIdx.x * blockDim.x + threadIdx.x; d < D; d += gridDim.x * blockDim.x)
        if (flip[d] < 1 || flip[d] > L - 1) atomicOr(bad, 1);
}

struct LevelLayout {
    size_t id, lv, total;
};

LevelLayout level_layout(int F, int L, int Wk)
{
    LevelLayout Ly;
    size_t off = 0;
    Ly.id = off; off = align_up(off + (size_t)F * Wk * 4, kAlign);
    Ly.lv = off; off = align_up(off + (size_t)L * Wk * 4, kAlign);
    Ly.total = off;
    return Ly;
}

constexpr int SMS = 152;   // a GB300: the lines below were measured on it, and no result depends on it
constexpr size_t FEW_SMEM = 220 * 1024, ENCODE_SMEM = 200 * 1024;   // most shared memory of a block; of staged rows

template <int NFW>
cudaError_t launch_count(const float *X, int64_t N, const hdc_levelid_model &m, uint32_t *H, int64_t slices, cudaStream_t st)
{
    auto k = levelid_count_kernel<NFW>;
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)count_smem<NFW>());
    if (e != cudaSuccess) return e;
    const int64_t tiles = (N + 31) / 32, share = std::max<int64_t>((NFW <= 8 ? 2 : 1) * SMS / slices, 1);
    k<<<dim3((unsigned)std::min(tiles, share), (unsigned)slices), CT, count_smem<NFW>(), st>>>(X, N, m.F, m.L, m.W, m.lo, m.scale,
                                                                                            m.id, m.level, H);
    return cudaGetLastError();
}

// The kernel of a query a thread, from both sides timed (us, this kernel / the
// rows' kernel; N * slices 32-query tiles are a round of the chip's warps for
// 38,912).  Below 30,000 the rows' kernel's shorter waves win (20,000 x 617 x
// 1,024: 181 / 205, 12,000: 144 / 134).  Every level costs 7 operations a
// feature word whatever its dims, so with many levels it takes more features
// (39,000 x 1,024 dims, 128 levels: 432 features ~232 / 215, 512: 231 / 284; 256:
// 143 / 134; 16 levels: 193 features 95 / 102, 256: 95 / 128), and the kernels
// come in 8, 12, 16, 20 and 25 words (257 features, 16 levels: 136 / 132).
bool use_count(int64_t N, int F, int L, int64_t slices)
{
    if (L > 128 || F > 800 || N * slices < 30000) return false;
    return L <= 32 ? F > 192 && (F <= 256 || F >= 272) : F >= 448;
}

size_t encode_smem(int F, int L) { return (size_t)(F + L) * LWC * 4; }

}  // namespace
}  // namespace hdc

using namespace hdc;

extern "C" hdc_status hdc_levelid_model_bytes(int32_t F, int32_t D, int32_t L, const hdc_approx_config *cfg,
                                              size_t *bytes)
{
    Perf p;
    if (!bytes || F <= 0 || D <= 0 || L < 2 || (cfg && cfg->struct_size < sizeof(hdc_approx_config)) ||
        !perf_of(D, cfg, &p))
        return HDC_ERR_INVALID_ARG;
    if (F >= 8 * 1024 || encode_smem(F, L) > ENCODE_SMEM) return HDC_ERR_UNSUPPORTED;
    *bytes = level_layout(F, L, words_for(p.Dk)).total;
    return HDC_OK;
}

extern "C" hdc_status hdc_levelid_prepare(const uint8_t *id_bits, const uint8_t *lo_bits, const uint8_t *hi_bits,
                                          const int32_t *flip, int32_t F, int32_t D, int32_t L, float x_lo,
                                          float x_hi, const hdc_approx_config *cfg, void *buf, size_t buf_bytes,
                                          int32_t *flip_error, hdc_levelid_model *out, hdc_stream_t stream)
{
    size_t need = 0;
    hdc_status s = hdc_levelid_model_bytes(F, D, L, cfg, &need);
    if (s != HDC_OK) return s;
    if (!id_bits || !lo_bits || !hi_bits || !flip || !out || !buf || ((uintptr_t)buf % kAlign) != 0 ||
        !(x_hi > x_lo) || !std::isfinite(x_lo) || !std::isfinite(x_hi))
        return HDC_ERR_INVALID_ARG;
    if (buf_bytes < need) return HDC_ERR_WORKSPACE;
    Perf p;
    perf_of(D, cfg, &p);
    const int Wk = words_for(p.Dk);
    const LevelLayout Ly = level_layout(F, L, Wk);
    cudaStream_t st = (cudaStream_t)stream;
    char *b = (char *)buf;
    if (flip_error) {
        if (cudaMemsetAsync(flip_error, 0, sizeof(int32_t), st) != cudaSuccess) return HDC_ERR_CUDA;
        flip_check_kernel<<<(D + 255) / 256 < 1024 ? (D + 255) / 256 : 1024, 256, 0, st>>>(flip, D, L, flip_error);
        if (cudaGetLastError() != cudaSuccess) return HDC_ERR_CUDA;
    }
    const int64_t n = (int64_t)(F + L) * Wk;
    levelid_prepare_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(
        id_bits, lo_bits, hi_bits, flip, F, L, (int64_t)D, p.s0, p.stride, p.Dk, Wk, (uint32_t *)(b + Ly.id),
        (uint32_t *)(b + Ly.lv));
    if (cudaGetLastError() != cudaSuccess) return HDC_ERR_CUDA;
    hdc_levelid_model m;
    memset(&m, 0, sizeof(m));
    m.struct_size = sizeof(m);
    m.F = F;
    m.D = D;
    m.Dk = (int32_t)p.Dk;
    m.L = L;
    m.W = Wk;
    m.lo = x_lo;
    m.scale = (float)((double)L / ((double)x_hi - (double)x_lo));
    m.id = (const uint32_t *)(b + Ly.id);
    m.level = (const uint32_t *)(b + Ly.lv);
    *out = m;
    return HDC_OK;
}

extern "C" hdc_status hdc_levelid_encode(const float *X, int64_t N, const hdc_levelid_model *m, uint32_t *H,
                                         hdc_stream_t stream)
{
    if (N < 0 || !m || m->struct_size < sizeof(hdc_levelid_model) || m->F <= 0 || m->L < 2 || m->Dk <= 0 ||
        m->W != words_for(m->Dk) || !m->id || !m->level || encode_smem(m->F, m->L) > ENCODE_SMEM || m->F >= 8 * 1024)
        return HDC_ERR_INVALID_ARG;
    if (N == 0) return HDC_OK;
    if (!X || !H) return HDC_ERR_INVALID_ARG;
    const cudaStream_t st = (cudaStream_t)stream;
    const int64_t slices = (m->W + LWC - 1) / LWC;
    if (slices > 65535) return HDC_ERR_UNSUPPORTED;
    const bool many = use_count(N, m->F, m->L, slices);
    if (many && (m->F <= 256   ? launch_count<8>(X, N, *m, H, slices, st)
                 : m->F <= 384 ? launch_count<12>(X, N, *m, H, slices, st)
                 : m->F <= 512 ? launch_count<16>(X, N, *m, H, slices, st)
                 : m->F <= 640 ? launch_count<20>(X, N, *m, H, slices, st)
                               : launch_count<25>(X, N, *m, H, slices, st)) != cudaSuccess)
        return HDC_ERR_CUDA;
    // one and four queries a warp where that is a wave of one block an SM
    for (int q1 = 1; q1 <= 4 && !many; q1 += 3) {
        const int64_t blocks = (N + LWARPS * q1 - 1) / (LWARPS * q1);
        const size_t smem = encode_smem(m->F, m->L) + (size_t)LWARPS * q1 * ((m->F + 3) / 4 * 4) * 4;
        if (blocks * slices > SMS || smem > FEW_SMEM || (((uintptr_t)m->id | (uintptr_t)m->level) & 15)) continue;
        auto k = hp_for(m->F) == 6 ? (q1 == 1 ? levelid_few_kernel<6, 1> : levelid_few_kernel<6, 4>)
                                   : (q1 == 1 ? levelid_few_kernel<9, 1> : levelid_few_kernel<9, 4>);
        if (allow_smem(k, FEW_SMEM) != cudaSuccess) return HDC_ERR_CUDA;
        k<<<dim3((unsigned)blocks, (unsigned)slices), LWARPS * 32, smem, st>>>(X, N, m->F, m->L, m->W, m->lo, m->scale, m->id,
                                                                              m->level, H);
        return cudaGetLastError() == cudaSuccess ? HDC_OK : HDC_ERR_CUDA;
    }
    const size_t smem = encode_smem(m->F, m->L) + LOFF_BYTES;
    // counter planes for floor(F / 16) (F < 8192: at most 9)
    auto k = hp_for(m->F) != 6 ? levelid_encode_kernel<9, false>
             : many            ? levelid_encode_kernel<6, true>
                               : levelid_encode_kernel<6, false>;
    if (allow_smem(k, ENCODE_SMEM + LOFF_BYTES) != cudaSuccess) return HDC_ERR_CUDA;
    // after the kernel above only what it left out: two blocks an SM, if any stay
    const int64_t blocks = (N + LQ - 1) / LQ;
    const dim3 grid((unsigned)(many ? std::min<int64_t>(blocks, (2 * SMS + slices - 1) / slices) : blocks), (unsigned)slices);
    k<<<grid, LWARPS * 32, smem, st>>>(X, N, m->F, m->L, m->W, m->lo, m->scale, m->id, m->level, H);
    return cudaGetLastError() == cudaSuccess ? HDC_OK : HDC_ERR_CUDA;
}
