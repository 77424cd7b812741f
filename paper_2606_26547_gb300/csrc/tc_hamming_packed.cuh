// Packed +-1 rows against small-integer class rows on the tensor cores: the
// Hamming arg-min of packed binary hypervectors (Sec. 4.1 Hamming distance
// and arg-min primitives) for up to 256 classes.
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
// Roles (19 warps):
//   warps 0-7   expand: a thread takes 256 dims (MT = 2: a row each) or 128
//               dims (MT = 1: a row's half) of every 256-dim tile from the
//               staged query words and writes them into its own TMEM lane
//               (tcgen05.st), double buffered; operand A of the MMAs;
//   warps 8-15  epilogue: D2 -> distances and arg-min, while the next unit's
//               tiles accumulate into the other D2 (R <= 64);
//   warp 16     TMA producer of the packed query words, 1,024 dims x MT x 128
//               rows per copy (whole 128-byte lines), a ring of HP_QB chunks;
//   warp 17     PRE: TMA producer of the class bytes (atoms of R rows x 128
//               dims) into a ring of p.nbs slots;
//   warp 18     MMA issuer.
// PRE: the class rows come already expanded (Cp rows of ldcs bytes, from
// launch_class_bytes into the caller's workspace).  Without it the expanding
// warps also expand the class words of every tile into two shared-memory
// buffers.
//
// Split rows: a batch of few units is given to clusters of p.S CTAs, each
// accumulating a contiguous part of the dims; the partial D2 are exchanged
// through distributed shared memory and the row groups of the unit are
// finished by the ranks in turn.
//
// TMEM (512 columns): D2 in columns 0..255 (MT x RS columns a buffer, RS = R
// rounded up to 32), the two query buffers of MT x 64 columns from 256.
// Every wait is bounded as in the encoder.
//
// What bounds it, and the form before: see launch_hamming_packed.
#pragma once
#include "tc_hamming.cuh"

namespace hdc {
namespace tc {

constexpr int HP_EXP = 256;                    // expanding threads (warps 0-7)
constexpr int HP_EPI0 = HP_EXP / 32;           // first of the eight epilogue warps
constexpr int HP_QPROD = 16, HP_BPROD = 17, HP_ISSUER = 18;
constexpr int HP_THREADS = 19 * 32;
constexpr int HP_CMAX = 256;
constexpr int HP_MAX_W = 4096;                 // words of a packed row (D <= 131072)
constexpr int HP_QB = 3;                       // query chunks in the ring
constexpr int HP_CHUNK = 4;                    // 256-dim tiles per query chunk (128 bytes of a row)
constexpr int HP_NBS_MAX = 16;                 // most class-atom slots
constexpr int HP_SMAX = 8;                     // most CTAs a unit's dims are split over
constexpr uint32_t HP_ACOL = 256;              // first TMEM column of the query buffers
// qfull[QB], qempty[QB], bfull[NBS], bempty[NBS], afull[2], aempty[2], d2full[2], d2empty[2], done
constexpr int HP_NUM_BARS = 2 * HP_QB + 2 * HP_NBS_MAX + 9;
constexpr int HP_TAIL = HP_NUM_BARS * 8 + 16 + 2 * HP_CMAX * 4;   // barriers, TMEM slot, abort flag, group counts

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

// 128 dims (four words) of a row into 32 TMEM columns of its lane.
__device__ __forceinline__ void hp_expand_tmem(uint32_t taddr, const uint4 w)
{
    const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
    uint32_t b[32];
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 8; j++) b[8 * i + j] = hp_signs(ws[i], j);
    hp_tmem_st32(taddr, b);
}

// 128 dims (four words) of class row r into its 128-byte row of a K atom
// (128-byte swizzle), zero outside the mask words.
__device__ __forceinline__ void hp_expand_row(uint8_t *atom, int r, const uint4 w, const uint4 m)
{
    uint8_t *row = atom + r * 128;
    const uint32_t ws[4] = {w.x, w.y, w.z, w.w}, ms[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
    for (int i = 0; i < 4; i++) {
        uint32_t b[8];
#pragma unroll
        for (int j = 0; j < 8; j++) b[j] = hp_signs(ws[i], j) & hp_mask(ms[i], j);
        *reinterpret_cast<uint4 *>(row + (((2 * i) ^ (r & 7)) * 16)) = make_uint4(b[0], b[1], b[2], b[3]);
        *reinterpret_cast<uint4 *>(row + (((2 * i + 1) ^ (r & 7)) * 16)) = make_uint4(b[4], b[5], b[6], b[7]);
    }
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
                 : "r"(a), "r"(rank)
                 : "memory");
    return v;
}

template <int MT, bool PRE>
__global__ void __launch_bounds__(HP_THREADS, 1)
    tc_hamming_packed_kernel(const HPParams p, const __grid_constant__ CUtensorMap tmQ,
                             const __grid_constant__ CUtensorMap tmC)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    constexpr int UROWS = MT * BM;                               // query rows of a unit
    constexpr int QCH = UROWS * 128;                             // bytes of a query chunk
    uint8_t *sQ = smem;
    uint8_t *sB = smem + hp_q_bytes(MT);                         // PRE: nbs atoms; else two tiles of two atoms
    const int atom_bytes = p.R * 128;
    uint32_t *smask = reinterpret_cast<uint32_t *>(sB + (size_t)(PRE ? p.nbs : 4) * atom_bytes);   // W words (not PRE)
    uint64_t *bars = reinterpret_cast<uint64_t *>(smask + (PRE ? 0 : ((p.W + 3) & ~3)));
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + HP_NUM_BARS);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    auto qfull = [&](int b) { return su32(bars + b); };
    auto qempty = [&](int b) { return su32(bars + HP_QB + b); };
    auto bfull = [&](int b) { return su32(bars + 2 * HP_QB + b); };
    auto bempty = [&](int b) { return su32(bars + 2 * HP_QB + HP_NBS_MAX + b); };
    constexpr int X = 2 * HP_QB + 2 * HP_NBS_MAX;
    auto afull = [&](int b) { return su32(bars + X + b); };
    auto aempty = [&](int b) { return su32(bars + X + 2 + b); };
    auto d2full = [&](int b) { return su32(bars + X + 4 + b); };
    auto d2empty = [&](int b) { return su32(bars + X + 6 + b); };
    const uint32_t done_bar = su32(bars + X + 8);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int RS = (p.R + 31) & ~31;                 // D2 columns of one 128-row tile
    const int ND2 = MT * RS <= 128 ? 2 : 1;          // D2 buffers
    const int64_t units = (p.N + UROWS - 1) / UROWS;
    const int S = p.S;
    const int rank = S > 1 ? (int)(blockIdx.x % S) : 0;
    const int64_t u0 = blockIdx.x / S, ustep = gridDim.x / S;
    const int chunks = (p.nt + HP_CHUNK - 1) / HP_CHUNK;
    const int ch0 = chunks * rank / S, ch1 = chunks * (rank + 1) / S;   // this rank's query chunks
    auto chunk_tiles = [&](int ch) { return min(HP_CHUNK, p.nt - ch * HP_CHUNK); };

    if (tid == 0) {
        for (int b = 0; b < HP_QB; b++) {
            mbar_init(qfull(b), 1);
            mbar_init(qempty(b), HP_EXP / 32);
        }
        for (int b = 0; b < HP_NBS_MAX; b++) {
            mbar_init(bfull(b), 1);
            mbar_init(bempty(b), 1);
        }
        for (int b = 0; b < 2; b++) {
            mbar_init(afull(b), HP_EXP / 32);
            mbar_init(aempty(b), 1);
            mbar_init(d2full(b), 1);
            mbar_init(d2empty(b), 4 * MT);
        }
        mbar_init(done_bar, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
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

    // Distances and arg-min of one row from its R dot products, read 32
    // columns at a time by `cols(j, v)`.
    auto finish = [&](int64_t row, auto cols) {
        const bool valid = row < p.N;
        int best = 0;
        float bd = -3.0e38f;   // largest dot = smallest distance; ascending c: lowest class on ties
        const bool vec = p.dists && p.C % 4 == 0 && (reinterpret_cast<uintptr_t>(p.dists) & 15) == 0;
        for (int j = 0; j * 32 < p.R; j++) {
            uint32_t v[32];
            cols(j, v);
#pragma unroll
            for (int i = 0; i < 32; i++) {
                const float d = __uint_as_float(v[i]);
                if (j * 32 + i < p.C && d > bd) { bd = d; best = j * 32 + i; }
            }
            if (p.dists && valid) {
                int32_t *o = p.dists + row * p.C + j * 32;
#pragma unroll
                for (int i = 0; i < 32; i++) v[i] = (uint32_t)((p.kept - (int)__uint_as_float(v[i])) / 2);
                if (vec) {
#pragma unroll
                    for (int i = 0; i < 32; i += 4)
                        if (j * 32 + i < p.C)
                            *reinterpret_cast<uint4 *>(o + i) = make_uint4(v[i], v[i + 1], v[i + 2], v[i + 3]);
                } else {
#pragma unroll
                    for (int i = 0; i < 32; i++)
                        if (j * 32 + i < p.C) o[i] = (int32_t)v[i];
                }
            }
        }
        if (valid) p.labels[row] = best;
    };

    if (warp == HP_ISSUER) {
        if (elect_one()) {  // ------------------------------ MMA issuer
            const uint32_t id = idesc_n<HDC_ENC_FP8_E4M3>(p.R);
            const uint64_t db0 = sdesc(su32(sB));
            int buf = 0, slot = 0, d2 = 0;
            uint32_t aph = 0, bph = 0, d2ph[2] = {0, 0};
            bool ab = false;
            for (int64_t u = u0; u < units && !ab; u += ustep) {
                if (!mbar_wait_fast(d2empty(d2), d2ph[d2] ^ 1, abort_flag)) { ab = true; break; }
                d2ph[d2] ^= 1;
                const uint32_t dcol = tmem + (uint32_t)(d2 * MT * RS);
                uint32_t accum = 0;
                for (int ch = ch0; ch < ch1 && !ab; ch++) {
                    const int ntl = chunk_tiles(ch);
                    for (int t = 0; t < ntl; t++) {
                        if (!mbar_wait_fast(afull(buf), aph, abort_flag)) { ab = true; break; }
                        const uint32_t acol = tmem + HP_ACOL + (uint32_t)(buf * MT * 64);
#pragma unroll
                        for (int a = 0; a < 2; a++) {   // two atoms of four 32-byte K steps
                            if (PRE && !mbar_wait_fast(bfull(slot), bph, abort_flag)) { ab = true; break; }
                            tc_fence_after();
                            const int at = PRE ? slot : buf * 2 + a;
                            const uint64_t db = db0 + (uint64_t)at * (uint64_t)(atom_bytes >> 4);
#pragma unroll
                            for (int m = 0; m < MT; m++)
#pragma unroll
                                for (int k = 0; k < 4; k++)
                                    h_mma_ts_fp8(dcol + (uint32_t)(m * RS), acol + (uint32_t)(m * 64 + a * 32 + 8 * k),
                                                 db + 2 * k, id, accum | (uint32_t)k);
                            accum = 1;
                            if (PRE) {
                                mma_commit(bempty(slot));
                                if (++slot == p.nbs) { slot = 0; bph ^= 1; }
                            }
                        }
                        if (ab) break;
                        mma_commit(aempty(buf));
                        if (++buf == 2) { buf = 0; aph ^= 1; }
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
                    const int n = isq ? 1 : 2 * chunk_tiles(ch);   // a query chunk, or the atoms of its tiles
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
        const int urow = MT == 2 ? tid : (tid & (BM - 1));      // row of the unit
        const int half = MT == 2 ? 0 : tid >> 7;                // MT = 1: this thread's 128 dims of a tile
        const uint32_t tlane = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t tcol = tmem + tlane + HP_ACOL + (uint32_t)(MT == 2 ? (warp >> 2) * 64 : half * 32);
        int buf = 0, qs = 0;
        uint32_t aph = 0, qph = 0;
        bool ab = false;
        // class words (not PRE): items i = tid and tid + 256, class i % R, half i / R of the tile
        auto class_words = [&](int i, int t) {
            const int c = i % p.R, wc = t * 8 + (i / p.R) * 4;
            return (i < 2 * p.R && c < p.C && wc < p.W)
                       ? __ldg(reinterpret_cast<const uint4 *>(p.cls + (int64_t)c * p.W + wc))
                       : make_uint4(0, 0, 0, 0);
        };
        for (int64_t u = u0; u < units && !ab; u += ustep) {
            uint4 cn0, cn1;
            if (!PRE) {
                cn0 = class_words(tid, ch0 * HP_CHUNK);
                cn1 = class_words(tid + HP_EXP, ch0 * HP_CHUNK);
            }
            for (int ch = ch0; ch < ch1 && !ab; ch++) {
                const bool okq = mbar_wait(qfull(qs), qph, abort_flag);
                if (!__all_sync(0xffffffffu, okq)) { ab = true; break; }
                const uint8_t *qrow = sQ + qs * QCH + urow * 128;
                const int ntl = chunk_tiles(ch);
                for (int tl = 0; tl < ntl; tl++) {
                    const int t = ch * HP_CHUNK + tl;
                    const uint4 w0 = *reinterpret_cast<const uint4 *>(qrow + (((tl * 2 + half) ^ (urow & 7)) << 4));
                    uint4 w1;
                    if (MT == 2) w1 = *reinterpret_cast<const uint4 *>(qrow + (((tl * 2 + 1) ^ (urow & 7)) << 4));
                    if (tl == ntl - 1) {   // the chunk's words are in registers: its slot may be refilled
                        __syncwarp();
                        if (lane == 0) mbar_arrive(qempty(qs));
                    }
                    const uint4 cw0 = cn0, cw1 = cn1;
                    if (!PRE && t + 1 < ch1 * HP_CHUNK && t + 1 < p.nt) {
                        cn0 = class_words(tid, t + 1);
                        cn1 = class_words(tid + HP_EXP, t + 1);
                    }
                    const bool oke = mbar_wait(aempty(buf), aph ^ 1, abort_flag);   // the MMAs of this buffer's last use
                    if (!__all_sync(0xffffffffu, oke)) { ab = true; break; }
                    tc_fence_after();
                    const uint32_t ta = tcol + (uint32_t)(buf * MT * 64);
                    hp_expand_tmem(ta, w0);
                    if (MT == 2) hp_expand_tmem(ta + 32, w1);
                    if (!PRE) {
#pragma unroll
                        for (int ii = 0; ii < 2; ii++) {
                            const int i = tid + ii * HP_EXP;
                            if (i < 2 * p.R) {
                                const int c = i % p.R, h = i / p.R, wc = t * 8 + h * 4;
                                const uint4 mc = (c < p.C && wc < p.W) ? *reinterpret_cast<const uint4 *>(smask + wc)
                                                                       : make_uint4(0, 0, 0, 0);
                                hp_expand_row(sB + (buf * 2 + h) * atom_bytes, c, ii ? cw1 : cw0, mc);
                            }
                        }
                        fence_async_smem();
                        __syncwarp();
                    }
                    h_tmem_st_wait();   // the query columns landed before the MMAs read them
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(afull(buf));
                    if (++buf == 2) { buf = 0; aph ^= 1; }
                }
                if (++qs == HP_QB) { qs = 0; qph ^= 1; }
            }
        }
    } else if (warp - HP_EPI0 < 4 * MT) {  // -------------- epilogue warps 8 .. 7 + 4 * MT
        const int e = warp - HP_EPI0;
        const uint32_t tlane = (uint32_t)((warp & 3) * 32) << 16;
        int d2 = 0;
        uint32_t d2ph = 0;
        for (int64_t u = u0; u < units; u += ustep) {
            const bool okd = mbar_wait(d2full(d2), d2ph, abort_flag);
            if (!__all_sync(0xffffffffu, okd)) break;
            tc_fence_after();
            const uint32_t dcol = tmem + tlane + (uint32_t)((d2 * MT + (e >> 2)) * RS);
            if (S == 1) {
                finish(u * UROWS + e * 32 + lane, [&](int j, uint32_t(&v)[32]) { tmem_ld32(dcol + (uint32_t)(j * 32), v); });
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
            finish(u0 * UROWS + e * 32 + lane, [&](int j, uint32_t(&v)[32]) {
#pragma unroll
                for (int i = 0; i < 32; i++) {
                    float s = 0.f;
                    if (j * 32 + i < p.R)
                        for (int k = 0; k < S; k++) s += hp_ld_cluster(base + (uint32_t)((j * 32 + i) * UROWS) * 4u, (uint32_t)k);
                    v[i] = __float_as_uint(s);
                }
            });
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
