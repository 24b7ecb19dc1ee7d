// trans_tc.cu -- Fuse (token slot), Mix and Trans of one pass on the graph
// path for bf16 refiners with more than 32 evaluated tokens (Sec. 4.1,
// Eq. fuse / mix / mlp), the two Trans products on tcgen05.
//
//   k_mix_c     per block and 32-channel slice: e_j = E'[x_{j-1}] for the
//               block's positions, c_k = Pc_k + e_k + sum_{j<k} L_kj e_j for
//               the positions the pass evaluates; c goes to cbuf (fp32, the
//               residual of Eq. mlp) and, rounded to bf16, to zpack (the
//               W_1 operand; the W_2 kernel later overwrites it with z)
//   k_trans_tc  D = A B^T on tcgen05, M = 128 evaluated tokens, N = 32
//               output units, K = 256 (W_1) or 512 (W_2):
//                 mode 1: A = bf16(c), B = W_1 rows; u = bf16(sigma(D)) to ubuf
//                 mode 2: A = u, B = W_2 rows; z = c + D to z_final (fp32, at
//                         the token's position) and bf16(z) to zpack (the
//                         Read's operand)
// Roles of k_trans_tc (192 threads): warp 0 TMA producer (one stage per
// K-chunk; the weight tiles before the dependency wait, the tokens after it),
// warp 1 TMEM allocator and MMA issuer, warps 2-5 epilogue (one TMEM lane
// quarter each).  Tiles whose first token is past the pass's count exit after
// the dependency wait, once their weight tiles have landed.  Both kernels are
// latency-bound: with the weights loaded before the wait, the residual beside the
// product and the call's parameters in shared memory a pass of 80 tokens takes
// 20.5 us through mix and Trans instead of 23.5.
#include "common.cuh"
#include "kernels.h"

namespace xp {

namespace {

constexpr int TT_BM = 128;                     // tokens (M)
constexpr int TT_BN = 32;                      // output units (N): many CTAs for a few token tiles
constexpr int TT_BK = 64;
constexpr int TT_STAGES = 8;                   // every K-chunk of W_2 (K = 512) has its own stage
constexpr uint32_t TT_A_STAGE = TT_BM * TT_BK * 2;    // 16 KB
constexpr uint32_t TT_B_STAGE = TT_BN * TT_BK * 2;    // 4 KB
constexpr uint32_t TT_STAGE = TT_A_STAGE + TT_B_STAGE;
constexpr uint32_t TT_IDESC = idesc_bf16(TT_BM, TT_BN);

struct TtShared {
    uint64_t full[TT_STAGES];
    uint64_t wfull, tfull;
    Params p;
    uint32_t tmem_base;
    int abort;
    int n;
};

}  // namespace

// K's chunks only: with K = 256 two CTAs fit an SM, so that the 256 CTAs of W_1 at
// 2048 tokens run in one wave (17.5 -> 11.7 us under ncu)
size_t trans_tc_smem(int K) { return 1024 + (size_t)(K / TT_BK) * TT_STAGE + sizeof(TtShared); }
const size_t kTransTcSmemBytes = trans_tc_smem(TT_STAGES * TT_BK);

// grid (8, b), 256 threads.  CTA `rank` of block s: channels [32 rank, +32).  A
// thread takes a channel pair of one position (two where the block has more
// than 16): its row of L and its Pc do not depend on the tokens and are
// requested before the gather, by 4-byte loads.  Latency-bound.
__global__ void __launch_bounds__(256) k_mix_c(const Params *__restrict__ pp)
{
    pdl_trigger();                     // the W_1 kernel may start its prologue
    __shared__ Params p;
    stage_params(&p, pp);
    __syncthreads();
    pdl_wait();                        // the previous pass (or the precompute) is complete
    const int rank = blockIdx.x, s = blockIdx.y, B = p.B;
    const SeqState st = p.st[s];
    if (!st.active) return;
    const int m = st.m, cnt = st.cnt, off = st.off;
    const int d0 = rank * 32;
    __shared__ __align__(8) float e[MAX_B][32];
    uint32_t lw[MAX_B - 1];
    float2 pc;
    auto load = [&](int i) {
        const int k = m + 1 + i / 16, d = d0 + 2 * (i % 16);
        const uint32_t *lp = reinterpret_cast<const uint32_t *>(p.Lpk + (size_t)(k * (k - 1) / 2) * RANK + d);
#pragma unroll
        for (int j = 0; j < MAX_B - 1; ++j)
            if (j < k) lw[j] = __ldg(lp + (size_t)j * (RANK / 2));
        pc = *reinterpret_cast<const float2 *>(p.Pc + ((size_t)s * B + k) * RANK + d);
    };
    int i = threadIdx.x;
    if (i < cnt * 16) load(i);
    for (int q = threadIdx.x; q < B * 32; q += blockDim.x) {
        const int j = q / 32, dd = q % 32;
        int x = j == 0 ? p.anchor[s] : p.tokens[(size_t)s * B + j - 1];
        if (x < 0 || x >= p.V) x = 0;   // reported by k_init
        e[j][dd] = p.Ep[(size_t)x * RANK + d0 + dd];
    }
    __syncthreads();
    uint16_t *cop = static_cast<uint16_t *>(p.zpack);
    while (i < cnt * 16) {
        const int t = i / 16, dd = 2 * (i % 16), k = m + 1 + t;
        const float2 ek = *reinterpret_cast<const float2 *>(&e[k][dd]);
        float a0 = pc.x + ek.x, a1 = pc.y + ek.y;
#pragma unroll
        for (int j = 0; j < MAX_B - 1; ++j)
            if (j < k) {
                const float2 ej = *reinterpret_cast<const float2 *>(&e[j][dd]);
                a0 = fmaf(__uint_as_float(lw[j] << 16), ej.x, a0);
                a1 = fmaf(__uint_as_float(lw[j] & 0xFFFF0000u), ej.y, a1);
            }
        const size_t o = (size_t)(off + t) * RANK + d0 + dd;
        *reinterpret_cast<float2 *>(p.cbuf + o) = make_float2(a0, a1);
        *reinterpret_cast<uint32_t *>(cop + o) = (uint32_t)f2bf(a0) | ((uint32_t)f2bf(a1) << 16);
        i += 256;
        if (i < cnt * 16) load(i);
    }
}

// grid (ceil(N / 128), units / 32), 192 threads, trans_tc_smem(K) bytes.
__global__ void __launch_bounds__(192, 1)
    k_trans_tc(const Params *__restrict__ pp, const __grid_constant__ CUtensorMap tmap_a,
               const __grid_constant__ CUtensorMap tmap_b, int K, int mode)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    TtShared &sh = *reinterpret_cast<TtShared *>(base + K / TT_BK * TT_STAGE);
    const Params &p = sh.p;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int t0 = blockIdx.x * TT_BM, n0 = blockIdx.y * TT_BN;
    const int nch = K / TT_BK;         // <= TT_STAGES
    pdl_trigger();                     // the next kernel may start its prologue
    if (threadIdx.x == 0) {
        for (int i = 0; i < TT_STAGES; ++i) mbar_init(&sh.full[i], 1);
        mbar_init(&sh.wfull, 1);
        mbar_init(&sh.tfull, 1);
        sh.abort = 0;
        fence_barrier_init();
        // the weights do not depend on the previous kernel: their tiles come first
        tma_prefetch_desc(&tmap_a);
        mbar_expect_tx(&sh.wfull, (uint32_t)nch * TT_B_STAGE);
        for (int c = 0; c < nch; ++c)
            tma_load_2d(base + c * TT_STAGE + TT_A_STAGE, &tmap_b, &sh.wfull, c * TT_BK, n0);
    }
    stage_params(&sh.p, pp);
    __syncwarp();                      // not every lane of warp 1 copied parameters
    if (warp == 1) { tmem_alloc(&sh.tmem_base, TT_BN); tmem_relinquish(); }
    __syncthreads();
    pdl_wait();                        // the operands of this pass are complete
    if (threadIdx.x == 0) sh.n = p.ctl[CTL_NACT];
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sh.tmem_base;
    volatile int *abort = &sh.abort;
    const int n = sh.n;
    const bool live = t0 < n;          // uniform over the CTA

    if (warp == 0) {
        if (lane == 0) {
            for (int c = 0; live && c < nch; ++c) {
                mbar_expect_tx(&sh.full[c], TT_A_STAGE);
                tma_load_2d(base + c * TT_STAGE, &tmap_a, &sh.full[c], c * TT_BK, t0);
            }
            // no copy may still be landing when the CTA leaves
            int dummy = 0;
            mbar_wait(&sh.wfull, 0, &dummy, 100000000ull);
            for (int c = 0; live && c < nch; ++c) mbar_wait(&sh.full[c], 0, &dummy, 100000000ull);
        }
    } else if (live && warp == 1) {
        if (lane == 0) {
            bool ok = mbar_wait(&sh.wfull, 0, abort);
            for (int c = 0; c < nch && ok; ++c) {
                if (!mbar_wait(&sh.full[c], 0, abort)) { ok = false; break; }
                tc_fence_after();
                const uint32_t a0 = smem_u32(base + c * TT_STAGE), b0 = a0 + TT_A_STAGE;
#pragma unroll
                for (int kk = 0; kk < TT_BK / 16; ++kk)
                    tc_mma_bf16(tmem, smem_desc_sw128(a0 + kk * 32), smem_desc_sw128(b0 + kk * 32), TT_IDESC,
                                (c | kk) != 0);
            }
            tc_commit(&sh.tfull);      // also when stopped: the epilogue must not hang
        }
    } else if (live && warp >= 2) {
        // epilogue: warp (quarter q = warp % 4) -> tokens 32 q .. +31 of the tile
        const int q = warp & 3;
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        const int t = t0 + q * 32 + lane;
        const bool valid = t < n;
        // mode 2: the token and its residual row are requested while the product runs
        int tok = 0;
        float4 cv[TT_BN / 4];
        if (mode == 2 && valid) {
            tok = p.act_tok[t];
            const float4 *cr = reinterpret_cast<const float4 *>(p.cbuf + (size_t)t * RANK + n0);
#pragma unroll
            for (int c = 0; c < TT_BN / 4; ++c) cv[c] = cr[c];
        }
        const bool got = mbar_wait_warp(&sh.tfull, 0, abort);
        if (got) {
            tc_fence_after();
            float *zf = p.z_final ? p.z_final : p.zbuf;
            const bool zal = (reinterpret_cast<uintptr_t>(zf) & 15) == 0;   // the caller's z_final: any 4-byte boundary
#pragma unroll
            for (int g = 0; g < TT_BN / 32; ++g) {
                float v[32];
                tmem_ld32(tmem + lane_base + g * 32, v);
                if (!valid) continue;
                const int col = n0 + g * 32;
                if (mode == 1) {
                    uint32_t w[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        w[j] = (uint32_t)f2bf(act_fn(p.act, v[2 * j])) |
                               ((uint32_t)f2bf(act_fn(p.act, v[2 * j + 1])) << 16);
                    uint4 *dst = reinterpret_cast<uint4 *>(p.ubuf + (size_t)t * 2 * RANK + col);
#pragma unroll
                    for (int c = 0; c < 4; ++c) dst[c] = make_uint4(w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
                } else {
                    float *zr = zf + (size_t)tok * RANK + col;
                    uint32_t w[16];
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        const float4 x = cv[8 * g + c];
                        const float4 z = make_float4(x.x + v[4 * c], x.y + v[4 * c + 1], x.z + v[4 * c + 2], x.w + v[4 * c + 3]);
                        if (zal) {
                            reinterpret_cast<float4 *>(zr)[c] = z;
                        } else {
                            zr[4 * c] = z.x;
                            zr[4 * c + 1] = z.y;
                            zr[4 * c + 2] = z.z;
                            zr[4 * c + 3] = z.w;
                        }
                        w[2 * c] = (uint32_t)f2bf(z.x) | ((uint32_t)f2bf(z.y) << 16);
                        w[2 * c + 1] = (uint32_t)f2bf(z.z) | ((uint32_t)f2bf(z.w) << 16);
                    }
                    uint4 *dst = reinterpret_cast<uint4 *>(static_cast<uint16_t *>(p.zpack) + (size_t)t * RANK + col);
#pragma unroll
                    for (int c = 0; c < 4; ++c) dst[c] = make_uint4(w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, TT_BN);
    }
    if (threadIdx.x == 0 && sh.abort) set_status(p.status, ST_TIMEOUT);
}

}  // namespace xp
