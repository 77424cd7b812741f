// HD-Clustering (Sec. 5.1): K-means over binary hypervectors, built from the
// classification kernels.  Per iteration:
//   assign   every point to the nearest cluster hypervector: Hamming over the
//            kept dims of the training similarity, arg-min (lowest index on
//            ties)                         -> launch_similarity (K4)
//   changes  points whose cluster differs from the previous iteration
//   update   every cluster hypervector = the bundle of its members (sign of
//            the int32 sum over all D; a cluster without members bundles to
//            zero, i.e. all +1)             -> hdc_train_epoch mode 0 (K5/K6)
// then a final assignment under the inference similarity's kept dims.  The
// two similarity ops are perforated independently, as the paper's tuner
// treats them.
//
// Few clusters and points (StepPlan): an iteration is two launches,
// assign_count_kernel and update_kernel.
#include <algorithm>

#include "hdc_internal.cuh"

namespace hdc {
namespace {

__global__ void count_changes_kernel(const int32_t *__restrict__ cur, const int32_t *__restrict__ prev, int64_t N,
                                     int first, int32_t *__restrict__ out)
{
    int n = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
        n += first || cur[i] != prev[i];
#pragma unroll
    for (int o = 16; o; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
    if ((threadIdx.x & 31) == 0 && n) atomicAdd(out, n);
}

// ---- an iteration in two launches ------------------------------------------
//
// The separate kernels (assign, changes, memset, histogram, scatter, count,
// reduce) take 37 us an iteration at 7,797 x 1,024 x 26, nearly all of it launch
// gaps and short chains of dependent memory accesses: the points are 1 MB.  Here
// a block keeps 64 points in shared memory, finds their clusters, and counts the
// members' bits of every cluster from the same copy; 10.5 us.  Counts leave as
// bit planes (plane p of a word: bit p of the 32 dims' counts), as many as the
// cluster's members in the block need.  What is left is two launches' latency
// and, per block, one trip each for the clusters, the counts and the planes.

constexpr int STEP_ROWS = 64;      // points of a block
constexpr int STEP_PLANES = 7;     // counts up to STEP_ROWS
constexpr int STEP_MAXK = 64;
constexpr int UPD_SLICES = 16;     // most warps of an update block, each a part of the runs
constexpr int CHIP_SMS = 152;       // a GB300; not asked for, so that size query and call always agree
constexpr size_t STEP_SMEM = 200 * 1024;   // most shared memory of an assignment block

// Lines of the route, from both sides timed (us an iteration, 2 / 7 launches): a
// block's planes are K W words a plane, so runs * K * W bounds the traffic
// (9,700 x 4,096 x 26, 506 K: 28 / 36; 5,000 x 6,000 x 36, 535 K: 40 / 37;
// 16,000 x 2,048 x 50, 800 K: 44 / 37), K * W the time of one block (500 x 6,000 x
// 50, 9,400: 38 / 37; 500 x 10,000 x 26, 8,320: 33 / 36), N * W the copies of the
// rows (9,700 x 6,000 x 16, 1.8 M: 29 / 34; 16,000 x 4,096 x 10, 2.0 M: 34 / 32;
// 9,700 x 10,000 x 4, 3.1 M: 34 / 31).  Eight threads a point while the blocks fit
// one to an SM, four in two resident blocks beyond (20,000 x 1,024 x 26: 25.5 /
// 21.5; 8,000: 10.5 / 13.6).
struct StepPlan {
    bool ok;
    int S;             // threads a point
    int chunks, cm;    // clusters in `chunks` passes of cm (8, 16, 24, 32)
    int words;         // staged words of a cluster hypervector: a multiple of 4 S
    int rows;          // shared-memory words from one point to the next: 16 mod 32
    int runs, slices;  // blocks of an assignment; warps of an update block
    size_t smem;
};

StepPlan step_plan(int64_t N, int W, int K)
{
    StepPlan p = {};
    if (N <= 0 || N > 16384 || K > STEP_MAXK || (int64_t)K * W > 9000 || N * W > 1850000)
        return p;
    p.runs = (int)((N + STEP_ROWS - 1) / STEP_ROWS);
    if ((int64_t)p.runs * K * W > 520000) return p;
    p.S = p.runs <= CHIP_SMS && W >= 32 ? 8 : 4;
    p.chunks = K > 32 ? 2 : 1;
    p.cm = ((K + p.chunks - 1) / p.chunks + 7) / 8 * 8;
    p.words = (W + 4 * p.S - 1) / (4 * p.S) * (4 * p.S);
    p.rows = (p.words + 31) / 32 * 32 + 16;
    p.smem = (size_t)(STEP_ROWS * p.rows + p.chunks * p.cm * p.words + p.words) * 4;
    // an update block of 16 warps while the chip holds them all at once
    const int64_t blocks = (int64_t)W / 4 * K;
    for (p.slices = UPD_SLICES; p.slices > 2 && blocks * p.slices > CHIP_SMS * 48; p.slices /= 2) {}
    p.ok = p.smem <= STEP_SMEM;
    return p;
}

__device__ __forceinline__ void cp16(void *dst, const void *src, bool on)
{
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    const int n = on ? 16 : 0;   // zero-filled when off
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(n));
}

// Block b: the points from 64 b.  S threads share a point: thread s takes
// the words 4 s .. 4 s + 3 of every 4 S, 16 bytes of the point and of each
// cluster hypervector at a time.  The differing bits of the four words pass two
// full adders per cluster before the carries are counted (hamming_csa_kernel).
// planes[((b K + c) 7 + p) W + w]; counts[c runs + b].
template <int CM, int S>
__global__ void __launch_bounds__(STEP_ROWS * S) assign_count_kernel(const uint32_t *__restrict__ H, int64_t N, int W, int K,
                                                              int chunks, int P, int Wp, int runs,
                                                              const uint32_t *__restrict__ cls, int masked, int64_t s0,
                                                              int64_t e0, int64_t stride, int32_t *__restrict__ lab,
                                                              int first, int32_t *__restrict__ changes,
                                                              uint32_t *__restrict__ planes, int32_t *__restrict__ counts)
{
    constexpr int ROWS = STEP_ROWS, T = ROWS * S;
    extern __shared__ __align__(16) uint32_t csm[];
    uint32_t *srow = csm, *scls = srow + ROWS * P, *smask = scls + chunks * CM * Wp;
    __shared__ int32_t s_cnt[STEP_MAXK], s_off[STEP_MAXK];
    __shared__ uint8_t s_idx[ROWS];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t n0 = (int64_t)blockIdx.x * ROWS;
    const int nr = (int)min((int64_t)ROWS, N - n0);
    // the points: constant over the iterations, so read ahead of the update
    const int q4 = (P - 16) / 4;
    for (int i = tid; i < ROWS * q4; i += T) {
        const int r = i / q4, c4 = (i % q4) * 4;
        const bool ok = r < nr && c4 < W;
        cp16(srow + r * P + c4, ok ? (const void *)(H + (n0 + r) * W + c4) : (const void *)H, ok);
    }
    for (int w = tid; w < Wp; w += T) {
        uint32_t m = 0xffffffffu;
        if (masked) {   // kept dims s0, s0 + stride, ... < e0 inside this word
            m = 0;
            const int64_t base = (int64_t)w * 32, lo = max(s0, base), hi = min(e0, base + 32);
            if (lo < hi) {
                const int64_t x = (lo - s0) % stride;
                for (int64_t d = x ? lo + (stride - x) : lo; d < hi; d += stride) m |= 1u << (d - base);
            }
        }
        smask[w] = m;
    }
    for (int i = tid; i < STEP_MAXK; i += T) s_cnt[i] = 0;
    early_wait(cls, lab);
    const int r = tid / S, s = tid % S;
    const bool own = s == 0 && r < nr;
    const int was = own && !first ? lab[n0 + r] : -1;
    const int KP = chunks * CM, k4 = Wp / 4;
    for (int i = tid; i < KP * k4; i += T) {
        const int c = i / k4, c4 = (i % k4) * 4;
        const bool ok = c < K && c4 < W;
        cp16(scls + c * Wp + c4, ok ? (const void *)(cls + (int64_t)c * W + c4) : (const void *)cls, ok);
    }
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    __syncthreads();

    int best = 0x7fffffff;   // distance * 64 + cluster: the lowest index on ties
    for (int cb = 0; cb < KP; cb += CM) {
        uint32_t ones[CM];
        int dist[CM];
#pragma unroll
        for (int c = 0; c < CM; c++) ones[c] = 0, dist[c] = 0;
        for (int w = 4 * s; w < Wp; w += 4 * S) {
            const uint4 q = *reinterpret_cast<const uint4 *>(srow + r * P + w);
            const uint4 m = *reinterpret_cast<const uint4 *>(smask + w);
            const uint32_t *cw = scls + cb * Wp + w;
#pragma unroll
            for (int c = 0; c < CM; c++) {
                const uint4 v = *reinterpret_cast<const uint4 *>(cw + c * Wp);
                const uint32_t x0 = (q.x ^ v.x) & m.x, x1 = (q.y ^ v.y) & m.y, x2 = (q.z ^ v.z) & m.z, x3 = (q.w ^ v.w) & m.w;
                uint32_t &a = ones[c];
                const uint32_t y0 = (a & x0) | (x1 & (a | x0));
                a ^= x0 ^ x1;
                const uint32_t y1 = (a & x2) | (x3 & (a | x2));
                a ^= x2 ^ x3;
                dist[c] += __popc(y0) + __popc(y1);
            }
        }
#pragma unroll
        for (int c = 0; c < CM; c++) dist[c] = 2 * dist[c] + __popc(ones[c]);
        // sums over the S threads; each ends with a quarter (S = 4) or an eighth
        // of the clusters
        int h[CM / 2], t[CM / 4];
#pragma unroll
        for (int i = 0; i < CM / 2; i++) {
            const int send = s & 1 ? dist[i] : dist[CM / 2 + i], keep = s & 1 ? dist[CM / 2 + i] : dist[i];
            h[i] = keep + __shfl_xor_sync(0xffffffffu, send, 1);
        }
#pragma unroll
        for (int i = 0; i < CM / 4; i++) {
            const int send = s & 2 ? h[i] : h[CM / 4 + i], keep = s & 2 ? h[CM / 4 + i] : h[i];
            t[i] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
        }
        int c0 = cb + (s & 1) * (CM / 2) + (s >> 1 & 1) * (CM / 4);
        if (S == 4) {
#pragma unroll
            for (int i = 0; i < CM / 4; i++)
                if (c0 + i < K) best = min(best, t[i] * STEP_MAXK + c0 + i);
        } else {
            c0 += (s >> 2 & 1) * (CM / 8);
#pragma unroll
            for (int i = 0; i < CM / 8; i++) {
                const int send = s & 4 ? t[i] : t[CM / 8 + i], keep = s & 4 ? t[CM / 8 + i] : t[i];
                const int e = keep + __shfl_xor_sync(0xffffffffu, send, 4);
                if (c0 + i < K) best = min(best, e * STEP_MAXK + c0 + i);
            }
        }
    }
#pragma unroll
    for (int o = 1; o < S; o <<= 1) best = min(best, __shfl_xor_sync(0xffffffffu, best, o));
    const int c = best & (STEP_MAXK - 1);
    int rank = 0, moved = 0;
    if (own) {
        moved = was != c;
        lab[n0 + r] = c;
        rank = atomicAdd(&s_cnt[c], 1);
    }
    moved = __syncthreads_count(moved);
    if (tid == 0 && changes && moved) atomicAdd(changes, moved);
    if (warp == 0) {   // first member of each cluster in s_idx: lane l owns clusters 2 l, 2 l + 1
        const int a = s_cnt[2 * lane], b = s_cnt[2 * lane + 1];
        int x = a + b;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        s_off[2 * lane] = x - a - b;
        s_off[2 * lane + 1] = x - b;
    }
    for (int i = tid; i < K; i += T) counts[(int64_t)i * runs + blockIdx.x] = s_cnt[i];
    __syncthreads();
    if (own) s_idx[s_off[c] + rank] = (uint8_t)r;
    __syncthreads();
    const int nch = (W + 31) / 32;
    for (int job = warp; job < K * nch; job += T / 32) {
        const int g = job / nch, w = job % nch * 32 + lane, n = s_cnt[g], i0 = s_off[g];
        if (n == 0) continue;
        const int bits = 32 - __clz(n);
        uint32_t pl[STEP_PLANES];
#pragma unroll
        for (int p = 0; p < STEP_PLANES; p++) pl[p] = 0;
        for (int i = 0; i < n; i += 4) {   // four members at a time, those past the end zero
            uint32_t x[4];
#pragma unroll
            for (int u = 0; u < 4; u++) x[u] = i + u < n ? srow[s_idx[i0 + i + u] * P + w] : 0u;
            const uint32_t y0 = (x[0] & x[1]) | (x[2] & (x[0] | x[1]));
            x[0] ^= x[1] ^ x[2];
            const uint32_t y1 = (x[0] & x[3]) | (pl[0] & (x[0] | x[3]));
            pl[0] ^= x[0] ^ x[3];
            uint32_t z = (y0 & y1) | (pl[1] & (y0 | y1));
            pl[1] ^= y0 ^ y1;
#pragma unroll
            for (int p = 2; p < STEP_PLANES; p++) {
                const uint32_t y = pl[p] & z;
                pl[p] ^= z;
                z = y;
            }
        }
        if (w < W) {
            uint32_t *dst = planes + (((int64_t)blockIdx.x * K + g) * STEP_PLANES) * W + w;
#pragma unroll
            for (int p = 0; p < STEP_PLANES; p++)
                if (p < bits) dst[(int64_t)p * W] = pl[p];
        }
    }
}

// Block (four words, cluster c): the runs' planes of its members summed (a
// thread: dims j, j + 8, j + 16, j + 24 of one word, the warps a part of the runs
// each), acc = members - 2 * set bits, cls = its sign.
__global__ void __launch_bounds__(32 * UPD_SLICES) update_kernel(const uint32_t *__restrict__ planes,
                                                                 const int32_t *__restrict__ counts, int W, int D, int K,
                                                                 int runs, int32_t *__restrict__ acc,
                                                                 uint32_t *__restrict__ cls)
{
    __shared__ int32_t s_sum[UPD_SLICES][5][32];
    const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5, slices = blockDim.x >> 5, j = lane & 7;
    const int c = blockIdx.y, w = blockIdx.x * 4 + (lane >> 3);   // W is a multiple of 4
    early_wait(planes, counts);
    const int32_t *cnt = counts + (int64_t)c * runs;
    // pairs of 16-bit sums: up to 64 for each of a warp's runs
    uint32_t lo = 0, hi = 0;
    int members = 0;
    for (int base = slice; base < runs; base += 32 * slices) {
        const int mine = base + lane * slices < runs ? __ldcg(cnt + base + lane * slices) : 0;
        const int m = min(32, (runs - base + slices - 1) / slices);
#pragma unroll 8
        for (int i = 0; i < m; i++) {
            const uint32_t *src = planes + (((int64_t)(base + i * slices) * K + c) * STEP_PLANES) * W + w;
            uint32_t x[3], v = 0;   // read whether there are as many or not: the counts are still on their way
#pragma unroll
            for (int p = 0; p < 3; p++) x[p] = __ldcg(src + (int64_t)p * W);
            const int n = __shfl_sync(0xffffffffu, mine, i);
#pragma unroll
            for (int p = 0; p < 3; p++) v += (((n >> p ? x[p] : 0u) >> j) & 0x01010101u) << p;
            for (int p = 3; n >> p; p++) v += ((__ldcg(src + (int64_t)p * W) >> j) & 0x01010101u) << p;
            lo += v & 0x00ff00ffu;
            hi += (v >> 8) & 0x00ff00ffu;
            members += n;
        }
    }
    int sum[5] = {(int)(lo & 0xffffu), (int)(hi & 0xffffu), (int)(lo >> 16), (int)(hi >> 16), members};
#pragma unroll
    for (int k = 0; k < 5; k++) s_sum[slice][k][lane] = sum[k];
    __syncthreads();
    if (slice != 0) return;
#pragma unroll
    for (int k = 0; k < 5; k++)
#pragma unroll
        for (int q = 1; q < UPD_SLICES; q++)
            if (q < slices) sum[k] += s_sum[q][k][lane];
    uint32_t bits = 0;
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const int d = w * 32 + j + 8 * k;
        if (d < D) {
            const int v = sum[4] - 2 * sum[k];
            acc[(int64_t)c * D + d] = v;
            bits |= (uint32_t)(v < 0) << (j + 8 * k);
        }
    }
    bits |= __shfl_xor_sync(0xffffffffu, bits, 1);
    bits |= __shfl_xor_sync(0xffffffffu, bits, 2);
    bits |= __shfl_xor_sync(0xffffffffu, bits, 4);
    if (j == 0) cls[(int64_t)c * W + w] = bits;
}

template <int S>
auto assign_count_of(int cm)
{
    return cm == 8 ? assign_count_kernel<8, S> : cm == 16 ? assign_count_kernel<16, S>
           : cm == 24 ? assign_count_kernel<24, S> : assign_count_kernel<32, S>;
}

// One iteration.  Only a launch that follows another of these starts early
// (what came before may still be writing H).
cudaError_t launch_step(const StepPlan &p, const uint32_t *H, int64_t N, int W, int D, int K, const Perf *mask, uint32_t *cls,
                        int32_t *acc, int32_t *lab, int first, int32_t *changes, uint32_t *planes, int32_t *counts,
                        cudaStream_t st)
{
    auto k = p.S == 4 ? assign_count_of<4>(p.cm) : assign_count_of<8>(p.cm);
    cudaError_t e = cudaSuccess;
    if (first) e = allow_smem(k, STEP_SMEM);
    if (e != cudaSuccess) return e;
    e = launch_early(k, dim3((unsigned)p.runs), (unsigned)(STEP_ROWS * p.S), p.smem, st, !first, H, N, W, K, p.chunks, p.rows,
                     p.words, p.runs, cls, mask ? 1 : 0, mask ? mask->s0 : 0, mask ? mask->e0 : 0, mask ? mask->stride : 1,
                     lab, first, changes, planes, counts);
    if (e != cudaSuccess) return e;
    return launch_early(update_kernel, dim3((unsigned)(W / 4), (unsigned)K), (unsigned)(32 * p.slices), 0, st, true, planes,
                        counts, W, D, K, p.runs, acc, cls);
}

struct ClusterLayout {
    size_t lab0, lab1, signs, train, planes, counts, total;
};

bool cluster_layout(int64_t N, int D, int K, ClusterLayout *L)
{
    size_t tb = 0;
    if (hdc_train_workspace_bytes(N, D, K, &tb) != HDC_OK) return false;
    size_t off = 0;
    L->lab0 = off;  off = align_up(off + (size_t)N * 4, kAlign);
    L->lab1 = off;  off = align_up(off + (size_t)N * 4, kAlign);
    // the cluster hypervectors expanded to bytes for the assignment (K > 16)
    L->signs = off; off = align_up(off + scratch_sign_bytes(K, words_for(D)), kAlign);
    L->train = off; off = align_up(off + tb, kAlign);
    const StepPlan p = step_plan(N, words_for(D), K);
    L->planes = off;
    if (p.ok) off = align_up(off + (size_t)p.runs * K * STEP_PLANES * words_for(D) * 4, kAlign);
    L->counts = off;
    if (p.ok) off = align_up(off + (size_t)p.runs * K * 4, kAlign);
    L->total = off;
    return true;
}

bool sim_ok(const hdc_approx_config *c)
{
    return !c || (c->struct_size >= sizeof(hdc_approx_config) && c->class_bits == 1);
}

// The kept dims of a similarity op (NULL when every dim of D is kept).
const Perf *perf_or_null(int64_t D, const hdc_approx_config *c, Perf *p)
{
    if (!c || !perf_of(D, c, p)) return nullptr;
    return (p->s0 == 0 && p->e0 == D && p->stride == 1) ? nullptr : p;
}

}  // namespace
}  // namespace hdc

using namespace hdc;

extern "C" hdc_status hdc_cluster_workspace_bytes(int64_t N, int32_t D, int32_t K, size_t *bytes)
{
    ClusterLayout L;
    if (!bytes || N < 0 || D <= 0 || K <= 0) return HDC_ERR_INVALID_ARG;
    if (N > kMaxTrainRows || K > kMaxTrainClasses) return HDC_ERR_UNSUPPORTED;
    if (!cluster_layout(N, D, K, &L)) return HDC_ERR_INVALID_ARG;
    *bytes = L.total;
    return HDC_OK;
}

extern "C" hdc_status hdc_cluster(const uint32_t *H, int64_t N, int32_t D, int32_t K, int32_t iters,
                                  const hdc_approx_config *train_sim, const hdc_approx_config *infer_sim,
                                  uint32_t *cls, int32_t *acc, int32_t *labels, int32_t *changes, void *ws,
                                  size_t ws_bytes, hdc_stream_t stream)
{
    if (N < 0 || D <= 0 || K <= 0 || iters < 0 || !cls || !acc || !labels || !sim_ok(train_sim) ||
        !sim_ok(infer_sim))
        return HDC_ERR_INVALID_ARG;
    // the perforations must keep at least one dim (checked by the Hamming entry on use)
    if (hdc_kept_dims(D, train_sim) <= 0 || hdc_kept_dims(D, infer_sim) <= 0) return HDC_ERR_INVALID_ARG;
    if (N > 0 && (!H || ((uintptr_t)H % 16) != 0)) return HDC_ERR_INVALID_ARG;
    if (((uintptr_t)cls % 16) != 0) return HDC_ERR_INVALID_ARG;
    if (N > kMaxTrainRows || K > kMaxTrainClasses) return HDC_ERR_UNSUPPORTED;
    ClusterLayout L;
    if (!cluster_layout(N, D, K, &L)) return HDC_ERR_INVALID_ARG;
    if (N > 0 && (!ws || ws_bytes < L.total || ((uintptr_t)ws % kAlign) != 0)) return HDC_ERR_WORKSPACE;
    cudaStream_t st = (cudaStream_t)stream;
    char *w = (char *)ws;
    int32_t *lab[2] = {(int32_t *)(w + L.lab0), (int32_t *)(w + L.lab1)};
    uint8_t *signs = scratch_sign_bytes(K, words_for(D)) ? (uint8_t *)(w + L.signs) : nullptr;
    const int W = words_for(D);
    Perf pt, pi;
    const Perf *ptrain = perf_or_null(D, train_sim, &pt), *pinfer = perf_or_null(D, infer_sim, &pi);
    if (changes && iters > 0 && cudaMemsetAsync(changes, 0, (size_t)iters * sizeof(int32_t), st) != cudaSuccess)
        return HDC_ERR_CUDA;
    if (N == 0) return HDC_OK;
    const StepPlan step = step_plan(N, W, K);
    for (int t = 0; step.ok && t < iters; t++)
        if (launch_step(step, H, N, W, D, K, ptrain, cls, acc, lab[0], t == 0, changes ? changes + t : nullptr,
                        (uint32_t *)(w + L.planes), (int32_t *)(w + L.counts), st) != cudaSuccess)
            return HDC_ERR_CUDA;
    for (int t = 0; !step.ok && t < iters; t++) {
        int32_t *cur = lab[t & 1], *prev = lab[(t + 1) & 1];
        if (launch_argmin_ws(H, N, cls, K, W, D, ptrain, cur, signs, st) != cudaSuccess) return HDC_ERR_CUDA;
        if (changes) {
            const int blocks = (int)std::min<int64_t>((N + 255) / 256, 4096);
            count_changes_kernel<<<blocks, 256, 0, st>>>(cur, prev, N, t == 0, changes + t);
            if (cudaGetLastError() != cudaSuccess) return HDC_ERR_CUDA;
        }
        hdc_status s = hdc_train_epoch(H, cur, N, D, K, 0, acc, cls, nullptr, w + L.train, L.planes - L.train,
                                       stream);
        if (s != HDC_OK) return s;
    }
    return launch_argmin_ws(H, N, cls, K, W, D, pinfer, labels, signs, st) == cudaSuccess ? HDC_OK : HDC_ERR_CUDA;
}
