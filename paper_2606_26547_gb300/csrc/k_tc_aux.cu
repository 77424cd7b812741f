// Auxiliary tensor-core kernels in a translation unit of their own (with
// its own device status word): the Hamming arg-min of packed hypervectors
// and the failure-detection self-test.


#include "tc_hamming_packed.cuh"

namespace hdc {

// Tensor map of E4M3 class bytes (`rows` rows of ldcs bytes, boxes of 128 bytes
// x `box` rows, 128-byte swizzle, zeros past the rows), defined with the other
// map builders.
bool make_class_sign_map(CUtensorMap *m, const uint8_t *signs, int ldcs, int rows, int box);
// Tensor map of packed rows (N rows of W words): boxes of 32 words x 128 rows,
// 128-byte swizzle, zeros past W and N.
bool make_packed_map(CUtensorMap *m, const uint32_t *Q, int W, int64_t N);
namespace tc {

// Failure-detection self-test: thread 0 waits, through the bounded-wait
// routine of the tensor-core kernels, on an mbarrier that nothing arrives
// on; the expiry records status 1 (timeout) in this unit's status word.
__global__ void __launch_bounds__(32, 1) wait_selftest_kernel(unsigned long long limit_ns)
{
    __shared__ __align__(8) uint64_t bar;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        mbar_init(su32(&bar), 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    if (threadIdx.x == 0) (void)mbar_wait(su32(&bar), 0, &abort_flag, limit_ns);
}

}  // namespace tc

bool hamming_packed_ok(int C, int W)
{
    return C > 0 && C <= tc::HP_CMAX && W > 0 && W <= tc::HP_MAX_W && W % 4 == 0;
}

int hamming_packed_ldcs(int W) { return (W + 7) / 8 * 256; }

namespace {
// Class words -> E4M3 bytes in the packed kernel's dim order, zero outside
// the kept dims: a thread writes the four dims j, j + 8, j + 16, j + 24 of one
// word, 32 bytes a word.
__global__ void class_bytes_kernel(const uint32_t *__restrict__ cls, int C, int W, int ldw, int64_t D, int64_t s0,
                                   int64_t e0, int64_t stride, uint32_t *__restrict__ out)
{
    // the packed kernel may be set up meanwhile (it waits for this one's end)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)C * ldw) return;
    const int c = (int)(i / ldw), x = (int)(i % ldw), w = x >> 3, j = x & 7;
    uint32_t v = 0;
    if (w < W)
        v = tc::hp_signs(__ldg(cls + (int64_t)c * W + w), j) & tc::hp_mask(tc::hp_word_mask(w, D, s0, e0, stride), j);
    out[i] = v;
}

int hp_sms()
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) !=
                                                     cudaSuccess || sms <= 0)
        sms = 152;
    return sms;
}

// Units (MT x 128 rows), CTAs per unit, and the estimate of one form's time.
// A split needs its clusters resident together: 8 * floor(16 / S) clusters of S
// CTAs up to six, 15 of seven or eight (one of the SM groups is smaller: the
// occupancy query's answer; 16 of eight took two waves, 26 us for 14).
struct HpPlan {
    int mt, S;
    int64_t units, cost;
};
bool hp_resident(int64_t units, int S, int sms) { return units * S <= sms && units <= (S > 6 ? 14 : 8 * (16 / S)); }

// Cosine and sweep: waves x 256-dim tiles a CTA x the tile's time (two row tiles
// 5, one 3); as many CTAs a unit as fit, which also share its row groups' scores.
HpPlan hp_plan_scores(int64_t N, int mt, int chunks, int sms)
{
    HpPlan pl = {mt, 1, (N + mt * tc::BM - 1) / (mt * tc::BM), 0};
    for (int S = 2; S <= tc::HP_SMAX && S <= chunks; S++)
        if (hp_resident(pl.units, S, sms)) pl.S = S;
    const int64_t waves = (pl.units * pl.S + sms - 1) / sms;
    pl.cost = waves * ((chunks + pl.S - 1) / pl.S) * (mt == 2 ? 5 : 3);
    return pl;
}

// Hamming: 10 ns a wave's 256-dim tiles and R-column epilogue, and a split's
// barriers and its reading of R sums of S ranks, 1 us and up: a fit to the forms
// forced on 55 .. 30,000 rows of 400 .. 8,000 dims, 20 .. 220 classes (1,418
// timings, 95 % within a tenth; the form chosen is 1.0005 times the best on
// average).  Splitting whenever the clusters fit took 1.2 times the best, and a
// sixth of those calls longer than the kernel before this one: 16,222 x 1,219 x
// 98 15.3 us in two CTAs a unit, 8.4 in one, 11.2 before; 500 x 1,380 x 112 12.9,
// 8.8, 12.1.
HpPlan hp_plan_hamming(int64_t N, int mt, int R, int nt, bool pre, int sms)
{
    HpPlan best = {mt, 1, (N + mt * tc::BM - 1) / (mt * tc::BM), 0};
    const int chunks = (nt + tc::HP_CHUNK - 1) / tc::HP_CHUNK;
    const int tile = pre ? (mt == 1 ? 42 : 54) + R / 20 : mt == 1 ? 67 + R / 6 : 87 + R * 3 / 10;
    for (int S = 1; S <= tc::HP_SMAX && S <= chunks; S++) {
        if (S > 1 && !hp_resident(best.units, S, sms)) continue;
        const int64_t waves = (best.units * S + sms - 1) / sms;
        const int part = (chunks + S - 1) / S * tc::HP_CHUNK, tiles = part < nt ? part : nt;
        int64_t cost = waves * ((int64_t)tiles * tile + (mt == 1 ? R : R * 5 / 4));
        if (S > 1) cost += mt == 1 ? 110 + R * (165 * S + 20) / 100 : 130 + R * (160 * S + 140) / 100;
        if (S == 1 || cost < best.cost) {
            best.S = S;
            best.cost = cost;
        }
    }
    return best;
}
// Chooses the form of a task whose sizes and epilogue `p` holds, and launches
// it: mq the packed rows, mc the class bytes (PRE).
template <bool PRE, int FIN>
cudaError_t launch_packed_rows(tc::HPParams &p, const CUtensorMap &mq, const CUtensorMap &mc, cudaStream_t st)
{
    const int sms = hp_sms(), chunks = (p.nt + tc::HP_CHUNK - 1) / tc::HP_CHUNK;
    auto plan = [&](int mt) {
        return FIN == tc::HP_HAMMING || FIN == tc::HP_FEW ? hp_plan_hamming(p.N, mt, p.R, p.nt, PRE, sms)
                                                          : hp_plan_scores(p.N, mt, chunks, sms);
    };
    HpPlan pl = plan(1);
    constexpr int MT = FIN == tc::HP_FEW ? 1 : 2;   // few rows are one tile
    if (MT == 2 && p.R <= 128) {
        const HpPlan p2 = plan(2);
        if (p2.cost < pl.cost) pl = p2;
    }
    p.S = pl.S;
    // shared memory: the query ring, the class atoms, barriers; at least 120 KB
    // so that no second CTA shares the SM and waits for its TMEM columns
    const size_t fixed = 1024 + tc::hp_q_bytes(pl.mt) + tc::hp_tail(pl.mt), atom = (size_t)p.R * 128;
    size_t nbs = (kMaxSmem - fixed) / atom;
    if (nbs > (size_t)tc::HP_NBS_MAX) nbs = tc::HP_NBS_MAX;
    p.nbs = (int)nbs;
    size_t smem = fixed + (PRE ? nbs * atom : tc::hp_nab(pl.mt, false) * atom + (size_t)((p.W + 3) & ~3) * 4);
    if (smem < 120 * 1024) smem = 120 * 1024;
    auto k = pl.mt == 2 ? tc::tc_hamming_packed_kernel<MT, PRE, FIN> : tc::tc_hamming_packed_kernel<1, PRE, FIN>;
    cudaError_t e = allow_smem(k, kMaxSmem);
    if (e != cudaSuccess) return e;
    const int64_t ctas = pl.units * pl.S;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)(pl.S > 1 || ctas < sms ? ctas : sms));
    lc.blockDim = dim3(tc::HP_THREADS);
    lc.dynamicSmemBytes = smem;
    lc.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = (unsigned)pl.S;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    lc.attrs = at;
    lc.numAttrs = pl.S > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&lc, k, p, mq, mc);
}

// The rows Q in launches whose row coordinates fit the copies' 32 bits, whole
// 256-row units each.
constexpr int64_t HP_LAUNCH_ROWS = 0x7fffff00;
template <bool PRE, int FIN>
cudaError_t launch_packed(const tc::HPParams &all, const uint32_t *Q, const CUtensorMap *mc, cudaStream_t st)
{
    cudaError_t e = cudaSuccess;
    for (int64_t r0 = 0; r0 < all.N && e == cudaSuccess; r0 += HP_LAUNCH_ROWS) {
        tc::HPParams p = all;
        p.N = all.N - r0 < HP_LAUNCH_ROWS ? all.N - r0 : HP_LAUNCH_ROWS;
        if (p.labels) p.labels += r0;
        if (p.dists) p.dists += r0 * p.C;
        if (p.scores) p.scores += r0 * p.C;
        if (p.y) p.y += r0;
        CUtensorMap mq;
        if (!make_packed_map(&mq, Q + r0 * p.W, p.W, p.N)) return cudaErrorInvalidValue;
        e = launch_packed_rows<PRE, FIN>(p, mq, mc ? *mc : mq, st);
    }
    return e;
}
}  // namespace

// Form of a call.  Two 128-row tiles a unit halve the class bytes streamed per
// row (R x D bytes a unit); one tile a unit fills the chip with half the rows
// and is the only form past 128 class rows (two D2 of 256 columns do not fit).
// hp_plan_hamming takes the faster.  Measured, calls
// with the workspace, the two-CTA form before (one tile a unit, its class tile
// copied inside the expand -> MMA chain, bit-transposing expansion, MMAs issued
// under a lane test) -> this one:
//   10^5 x 16,384 dims: 100 classes 234 -> 136 us, 256 classes 396 -> 240
//   10^6 x 1,024 dims:  64 classes 185 -> 84 us, 200 classes 447 -> 234
// and without it (classes expanded per tile) 100 classes 365 -> 237 us, 26 ones 195.
cudaError_t launch_hamming_packed(const uint32_t *Q, int64_t N, const uint32_t *cls, int C, int W, int64_t D,
                                  int64_t s0, int64_t e0, int64_t stride, int32_t *labels, int32_t *dists,
                                  cudaStream_t st, uint8_t *signs)
{
    if (N <= 0) return cudaSuccess;
    if (!hamming_packed_ok(C, W) || stride < 1) return cudaErrorNotSupported;
    const int ldcs = hamming_packed_ldcs(W), R = (C + 15) / 16 * 16;
    CUtensorMap mc;
    if (signs) {   // the classes once into `signs`, zero outside the kept dims
        const int64_t n = (int64_t)C * (ldcs / 4);
        class_bytes_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(cls, C, W, ldcs / 4, D, s0, e0, stride,
                                                                        reinterpret_cast<uint32_t *>(signs));
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        if (!make_class_sign_map(&mc, signs, ldcs, C, R)) return cudaErrorInvalidValue;
    }
    tc::HPParams p = {};
    p.cls = cls;
    p.N = N;
    p.W = W;
    p.C = C;
    p.R = R;
    p.nt = (W + 7) / 8;
    p.D = D;
    p.s0 = s0;
    p.e0 = e0;
    p.stride = stride;
    const int64_t end = e0 < D ? e0 : D;
    p.kept = end > s0 ? (int)((end - s0 + stride - 1) / stride) : 0;
    p.labels = labels;
    p.dists = dists;
    if (dists && C % 4 != 0 && N <= 64)
        return signs ? launch_packed<true, tc::HP_FEW>(p, Q, &mc, st) : launch_packed<false, tc::HP_FEW>(p, Q, nullptr, st);
    return signs ? launch_packed<true, tc::HP_HAMMING>(p, Q, &mc, st) : launch_packed<false, tc::HP_HAMMING>(p, Q, nullptr, st);
}

cudaError_t launch_packed_cosine(const uint32_t *Q, int64_t N, int W, const uint8_t *vals, int C, int P,
                                 const double *cnorm, int32_t *labels, double *scores, cudaStream_t st)
{
    if (N <= 0) return cudaSuccess;
    const int rows = C * P, R = (rows + 15) / 16 * 16, ld = hamming_packed_ldcs(W);
    if (!hamming_packed_ok(rows, W) || P < 1 || P > 2) return cudaErrorNotSupported;
    CUtensorMap mc;
    if (!make_class_sign_map(&mc, vals, ld, rows, R)) return cudaErrorInvalidValue;
    tc::HPParams p = {};
    p.N = N;
    p.W = W;
    p.C = C;
    p.R = R;
    p.nt = (W + 7) / 8;
    p.P = P;
    p.cnorm = cnorm;
    p.labels = labels;
    p.scores = scores;
    return launch_packed<true, tc::HP_COSINE>(p, Q, &mc, st);
}

cudaError_t launch_packed_sweep(const PackedSweep &a, cudaStream_t st)
{
    if (a.N <= 0 || a.ncfg <= 0) return cudaSuccess;
    tc::HPParams p = {};
    int rows = 0;
    for (int i = 0; i < a.ncfg; i++) {
        p.cfg_p[i] = a.digits[i];
        p.cfg_k[i] = a.out[i];
        p.cfg_col[i] = (uint16_t)rows;
        rows += a.C * (a.digits[i] ? a.digits[i] : 1);
    }
    if (a.ncfg > tc::HP_MAXCFG || !hamming_packed_ok(rows, a.W)) return cudaErrorNotSupported;
    const int R = (rows + 15) / 16 * 16;
    CUtensorMap mc;
    if (!make_class_sign_map(&mc, a.vals, hamming_packed_ldcs(a.W), rows, R)) return cudaErrorInvalidValue;
    p.N = a.N;
    p.W = a.W;
    p.C = a.C;
    p.R = R;
    p.nt = (a.W + 7) / 8;
    p.ncfg = a.ncfg;
    p.sumsq = a.sumsq;
    p.y = a.y;
    p.correct = a.correct;
    p.labels = a.labels;
    p.ldl = a.N;
    return launch_packed<true, tc::HP_SWEEP>(p, a.H, &mc, st);
}

cudaError_t launch_wait_selftest(unsigned long long limit_ns, cudaStream_t st)
{
    tc::wait_selftest_kernel<<<1, 32, 0, st>>>(limit_ns);
    return cudaGetLastError();
}

cudaError_t tc_aux_read_status(cudaStream_t st, int *status) { return tc::read_status(st, status); }

}  // namespace hdc
