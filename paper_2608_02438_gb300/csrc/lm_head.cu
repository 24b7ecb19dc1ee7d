// lm_head.cu -- the drafter's base logits s = W_lm h (Sec. 4.1, Fig. 2a: the
// target-sized LM head that produces s_k before the refiner) with Algorithm
// 1's Y^(0) = argmax_v s_k,v fused into the epilogue.
//
// GEMM view: D[v, t] = W_lm[v, :] . h[t, :], M = MT tiles of 128 vocabulary
// rows (the weight stream, 1.245 GB at the Qwen3-8B shape), N = NT tokens (a
// chunk of the N hidden states), K = H.  Vocabulary rows sit in TMEM lanes, so
// the stores of s are runs of 64 bytes per token.  Up to 16 chunks at a time share
// the CTAs (LmWork), so that the CTAs of an item read the same rows of W_lm at about
// the same time: one read from HBM, the others from L2.
//
// Tiles by N (lm_shape): up to 32 tokens NT = 32, up to 128 NT = 128 (both
// HBM-bound on W_lm: the smaller the token part of a ring stage, the more of W_lm
// is in flight; 83 tokens 204 us against 236 in a 256-token chunk);
// beyond, NT = 256, where both operands come from L2 and tensor time and the
// L2-to-SM stream compete: MT = 2 loads 64 KB per 256 x 256 x 64 product instead
// of 48 KB per 128 x 256 x 64, at the price of a single accumulator (the epilogue is
// not overlapped).  Measured at the Qwen3-8B shape, MT = 2 / MT = 1 / MT = 1 and
// whole chunks one after the other, us: 129 tokens 215 / 216 / 216, 160 220 / 225 /
// 225, 256 255 / 255 / 256, 300 410 / 395 / 466, 384 393 / 415 / 483, 512 445 / 454 /
// 540, 1024 880 / 905 / 1065, 2048 1655 / 1740 / 2110 (512 without the stores of s:
// 433).  MT = 1 remains where MT = 2 would leave fewer than two items per CTA.
//
// Roles (32 (2 + 4 MT) threads):
//   warp 0     TMA producer: per K-chunk of 64, a 128 MT x 64 box of W_lm and an
//              NT x 64 box of h (rows past V or N read as zero), into a ring
//   warp 1     TMEM allocator and tcgen05.mma issuer (one thread); two
//              accumulators of MT NT columns where TMEM holds them, so that the
//              epilogue of one item overlaps the MMAs of the next
//   the others epilogue, 4 warps per 128-row tile: tcgen05.ld of 32 token columns
//              of its lane quarter, rounding to bf16 (the stored s), the stores of
//              s, and per token the running argmax over the rows this warp has
//              seen in the current chunk (a 32 x 32 bf16 transpose through shared
//              memory, so that lane t reduces token t)
// Every CTA leaves one (max, id) partial per token of its chunks; the second
// kernel combines the partials of each token (ties: smallest id).
#include "train_common.cuh"
#include "kernels.h"
#include "lm_work.h"

namespace xp {

namespace {

constexpr int LM_BM = 128;
constexpr int LM_BK = 64;

template <int NT, int MT>
struct LmShape {
    static constexpr int EPI_WARPS = 4 * MT;
    static constexpr int THREADS = 32 * (2 + EPI_WARPS);
    static constexpr uint32_t A_TILE = LM_BM * LM_BK * 2;      // 16 KB: 128 rows of W_lm
    static constexpr uint32_t A_STAGE = MT * A_TILE;
    static constexpr uint32_t STAGE = A_STAGE + NT * LM_BK * 2;
    static constexpr int STAGES = NT <= 32 ? 8 : (NT <= 128 ? 6 : (MT == 1 ? 4 : 3));
    static constexpr int NBUF = 2 * MT * NT <= 512 ? 2 : 1;    // accumulators
    static constexpr uint32_t TMEM_COLS = NBUF * MT * NT < 32 ? 32 : NBUF * MT * NT;   // a power of two
    static constexpr uint32_t IDESC = idesc_bf16(LM_BM, NT);
    static constexpr size_t TILE_BYTES = EPI_WARPS * 32 * 34 * 2;     // per-warp transposes
    static constexpr size_t BEST_BYTES = EPI_WARPS * NT * 8;          // per-warp running maxima of a chunk
    static constexpr size_t SCRATCH = TILE_BYTES + BEST_BYTES;
    static constexpr size_t SMEM = 1024 + (size_t)STAGES * STAGE + SCRATCH + 256;
};

struct LmBars {
    uint64_t full[8], empty[8];
    uint64_t tfull[2], tempty[2];
    uint64_t drain;
    uint32_t tmem_base;
    int abort;
};
static_assert(sizeof(LmBars) <= 256, "barriers");
static_assert(LmShape<32, 1>::SMEM <= 232448 && LmShape<128, 1>::SMEM <= 232448 && LmShape<256, 1>::SMEM <= 232448 &&
                  LmShape<256, 2>::SMEM <= 232448,
              "shared memory");

__device__ __forceinline__ bool better(float v, int i, float bv, int bi) { return v > bv || (v == bv && i < bi); }

}  // namespace

// grid G <= NC x items (every CTA has an item), LmShape::THREADS threads, LmShape::SMEM bytes.
template <int NT, int MT>
__device__ __forceinline__ void lm_head_body(const CUtensorMap &tmap_w, const CUtensorMap &tmap_h, int V, int H, int N,
                                             uint16_t *s_out, Partial *part, int32_t *status)
{
    using Sh = LmShape<NT, MT>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *scratch = base + Sh::STAGES * Sh::STAGE;
    LmBars &sh = *reinterpret_cast<LmBars *>(scratch + Sh::SCRATCH);
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int G = gridDim.x;
    const int NI = (V + MT * LM_BM - 1) / (MT * LM_BM), NC = (N + NT - 1) / NT, KCH = (H + LM_BK - 1) / LM_BK;
    const LmWork wk(blockIdx.x, G, NC);

    if (threadIdx.x == 0) {
        for (int i = 0; i < Sh::STAGES; ++i) { mbar_init(&sh.full[i], 1); mbar_init(&sh.empty[i], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&sh.tfull[i], 1); mbar_init(&sh.tempty[i], Sh::EPI_WARPS); }
        mbar_init(&sh.drain, 1);
        sh.abort = 0;
        fence_barrier_init();
    }
    if (warp == 1) { tmem_alloc(&sh.tmem_base, Sh::TMEM_COLS); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sh.tmem_base;
    volatile int *abort = &sh.abort;

    if (warp == 0) {
        // ------------------------------------------------------- producer
        if (lane == 0) {
            tma_prefetch_desc(&tmap_w);
            tma_prefetch_desc(&tmap_h);
            // W_lm: read once by one chunk, else again by the other chunks' CTAs; h: by every item
            const uint64_t pw = NC == 1 ? policy_evict_first() : policy_evict_normal(), ph = policy_evict_last();
            int stage = 0;
            uint32_t phase = 0, pending = 0, pend_par = 0;
            bool ok = true;
            for (int gr = 0; gr < wk.groups && ok; ++gr) {
                const int c = wk.chunk(gr), step = wk.step(gr);
                for (int it = wk.first(gr); it < NI && ok; it += step)
                    for (int kc = 0; kc < KCH; ++kc) {
                        if (!mbar_wait(&sh.empty[stage], phase ^ 1, abort)) { ok = false; break; }
                        uint8_t *dst = base + stage * Sh::STAGE;
                        mbar_expect_tx(&sh.full[stage], Sh::STAGE);
                        tma_load_2d_hint(dst, &tmap_w, &sh.full[stage], kc * LM_BK, it * MT * LM_BM, pw);
                        tma_load_2d_hint(dst + Sh::A_STAGE, &tmap_h, &sh.full[stage], kc * LM_BK, c * NT, ph);
                        pending |= 1u << stage;
                        pend_par = (pend_par & ~(1u << stage)) | (phase << stage);
                        if (++stage == Sh::STAGES) { stage = 0; phase ^= 1; }
                    }
            }
            // no copy may still be landing when the CTA leaves
            int dummy = 0;
            for (int st = 0; st < Sh::STAGES; ++st)
                if (pending & (1u << st)) mbar_wait(&sh.full[st], (pend_par >> st) & 1, &dummy, 100000000ull);
        }
    } else if (warp == 1) {
        // ---------------------------------------------------- MMA issuer
        if (lane == 0) {
            // descriptors formed once, advanced per MMA
            const uint64_t desc0 = smem_desc_sw128(smem_u32(base));
            int stage = 0, t = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int gr = 0; gr < wk.groups && ok; ++gr) {
                const int step = wk.step(gr);
                for (int it = wk.first(gr); it < NI && ok; it += step, ++t) {
                    const int buf = t % Sh::NBUF;
                    if (!mbar_wait(&sh.tempty[buf], ((t / Sh::NBUF) & 1) ^ 1, abort)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t d = tmem + buf * MT * NT;
                    for (int kc = 0; kc < KCH; ++kc) {
                        if (!mbar_wait(&sh.full[stage], phase, abort)) { ok = false; break; }
                        tc_fence_after();
                        const uint64_t ad = smem_desc_advance(desc0, stage * Sh::STAGE), bd = smem_desc_advance(ad, Sh::A_STAGE);
#pragma unroll
                        for (int m = 0; m < MT; ++m)
#pragma unroll
                            for (int kk = 0; kk < LM_BK / 16; ++kk)
                                tc_mma_bf16(d + m * NT, smem_desc_advance(ad, m * Sh::A_TILE + kk * 32),
                                            smem_desc_advance(bd, kk * 32), Sh::IDESC, (kc | kk) != 0);
                        tc_commit(&sh.empty[stage]);
                        if (++stage == Sh::STAGES) { stage = 0; phase ^= 1; }
                    }
                    if (ok) tc_commit(&sh.tfull[buf]);
                }
            }
            tc_commit(&sh.drain);
            int dummy = 0;
            mbar_wait(&sh.drain, 0, &dummy, 100000000ull);
        }
    } else {
        // ------------------------------------------------------ epilogue
        const int ew = warp - 2, q = warp & 3, m = ew >> 2;
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        uint16_t (*tp)[34] = reinterpret_cast<uint16_t (*)[34]>(scratch + ew * (32 * 34 * 2));
        float2 *best = reinterpret_cast<float2 *>(scratch + Sh::TILE_BYTES);   // [warp][NT] (value, id bits)
        int t = 0;
        bool got = true;
        for (int gr = 0; gr < wk.groups && got; ++gr) {
            const int c = wk.chunk(gr), slot = wk.first(gr), step = wk.step(gr);
#pragma unroll 1
            for (int g = 0; g < NT / 32; ++g)
                best[ew * NT + g * 32 + lane] = make_float2(-INFINITY, __int_as_float(0x7fffffff));
            for (int it = slot; it < NI && got; it += step, ++t) {
                const int buf = t % Sh::NBUF;
                got = mbar_wait_warp(&sh.tfull[buf], (t / Sh::NBUF) & 1, abort);
                tc_fence_after();
                const int row0 = (it * MT + m) * LM_BM + q * 32, row = row0 + lane;   // this thread's vocabulary row
#pragma unroll 1
                for (int g = 0; g < NT / 32; ++g) {
                    if (!got) break;
                    __syncwarp();
                    float v[32];
                    tmem_ld32(tmem + lane_base + (buf * MT + m) * NT + g * 32, v);
                    const int tok0 = c * NT + g * 32;
                    if (tok0 >= N) break;                                // padding tokens
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const uint16_t b = f2bf(v[j]);
                        if (s_out && row < V && tok0 + j < N) s_out[(size_t)(tok0 + j) * V + row] = b;
                        tp[j][lane] = row < V ? b : (uint16_t)0xFF80;    // [token][row of the quarter], -inf past V
                    }
                    __syncwarp();
                    // lane j: token tok0 + j over this quarter's 32 rows (ascending ids)
                    float mx = -INFINITY;
                    int mi = 0x7fffffff;
#pragma unroll
                    for (int rr = 0; rr < 16; ++rr) {
                        const uint32_t w = *reinterpret_cast<const uint32_t *>(&tp[lane][2 * rr]);
                        const float lo = __uint_as_float(w << 16), hi = __uint_as_float(w & 0xFFFF0000u);
                        if (lo > mx) { mx = lo; mi = row0 + 2 * rr; }
                        if (hi > mx) { mx = hi; mi = row0 + 2 * rr + 1; }
                    }
                    float2 &b = best[ew * NT + g * 32 + lane];             // this lane's own slot
                    if (better(mx, mi, b.x, __float_as_int(b.y))) b = make_float2(mx, __int_as_float(mi));
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.tempty[buf]);
            }
            // the chunk is done in this CTA: its partial per token
            if (warps_bar_or<32 * Sh::EPI_WARPS>(!got)) break;
            for (int j = threadIdx.x - 64; j < NT; j += Sh::EPI_WARPS * 32) {
                const int tok = c * NT + j;
                if (tok < N) {
                    float2 a = best[j];
                    for (int w = 1; w < Sh::EPI_WARPS; ++w) {
                        const float2 b = best[w * NT + j];
                        if (better(b.x, __float_as_int(b.y), a.x, __float_as_int(a.y))) a = b;
                    }
                    part[(size_t)tok * G + slot] = Partial{a.x, __float_as_int(a.y), 0.0f, 0.0f};
                }
            }
            warps_bar<32 * Sh::EPI_WARPS>();
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, Sh::TMEM_COLS);
    }
    if (threadIdx.x == 0 && sh.abort) set_status(status, ST_TIMEOUT);
    pdl_trigger();
}

// grid ceil(N / 8), 256 threads: warp w combines the partials of token
// 8 blockIdx.x + w (ties: the smallest id); G, NT as the product was launched.
__global__ void __launch_bounds__(256) k_lm_head_argmax(const Partial *part, int G, int NT, int N, int32_t *argmax_out)
{
    pdl_wait();
    const int tok = blockIdx.x * 8 + threadIdx.x / 32, lane = threadIdx.x % 32;
    if (tok >= N) return;
    const int NC = (N + NT - 1) / NT, c = tok / NT;
    const int slots = LmWork(0, G, NC).slots(c);                       // CTAs that worked on the token's chunk
    float m = -INFINITY;
    int mi = 0x7fffffff;
    for (int s = lane; s < slots; s += 32) {
        const Partial a = part[(size_t)tok * G + s];
        if (better(a.best, a.idx, m, mi)) { m = a.best; mi = a.idx; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float om = __shfl_xor_sync(0xffffffffu, m, o);
        const int oi = __shfl_xor_sync(0xffffffffu, mi, o);
        if (better(om, oi, m, mi)) { m = om; mi = oi; }
    }
    if (lane == 0) argmax_out[tok] = mi;
}

#define XP_LM_HEAD(name, NT, MT)                                                                                   \
    __global__ void __launch_bounds__(LmShape<NT, MT>::THREADS, 1)                                                 \
        name(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_h, int V, int H, \
             int N, uint16_t *s_out, Partial *part, int32_t *status)                                               \
    {                                                                                                              \
        lm_head_body<NT, MT>(tmap_w, tmap_h, V, H, N, s_out, part, status);                                        \
    }
XP_LM_HEAD(k_lm_head32, 32, 1)
XP_LM_HEAD(k_lm_head128, 128, 1)
XP_LM_HEAD(k_lm_head256, 256, 1)
XP_LM_HEAD(k_lm_head256x2, 256, 2)
#undef XP_LM_HEAD

template <int NT, int MT> static LmKernel lm_kernel(LmKernelFn fn)
{
    return LmKernel{fn, NT, MT, LmShape<NT, MT>::THREADS, LmShape<NT, MT>::SMEM};
}
const LmKernel kLmHeads[4] = {lm_kernel<32, 1>(k_lm_head32), lm_kernel<128, 1>(k_lm_head128),
                              lm_kernel<256, 1>(k_lm_head256), lm_kernel<256, 2>(k_lm_head256x2)};

}  // namespace xp
