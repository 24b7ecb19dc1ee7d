// train_read.cu -- the Read GEMM of the refiner training step (Sec. 4.3) on
// tcgen05, fused with the softmax / total-variation arithmetic of the loss
// L(p) = sum_k w_k [a_ce (-log p_k(y*_k)) + a_l1 |p_k - p^t_k|_1]
// and of its gradient.  The logits l = s + W_r z of all rows are recomputed by
// every pass instead of being stored (N x V floats would cost more HBM traffic
// than re-reading s and t).
//
// Rows: the refiner runs twice per position (teacher-forced inputs and the
// consistency inputs argmax s); a 128-row tile holds 64 positions, rows 0-63
// the teacher-forced forward and rows 64-127 the consistency forward of the
// same positions, so that one s / t tile of those 64 positions serves both.
//
// k_train_tok -- token-major: D[row, v] = z_row . W_r[v], M = 128 rows, N = 128
// vocabulary ids in TR_STATS, 64 in TR_TV and TR_DZ, K = r.  CTA (split, tile) takes one row tile and a
// contiguous range of vocabulary tiles.  The row tile Z sits in tensor memory
// as the A operand (with N = 64, re-reading a 4 KB A block from shared memory
// for every MMA would cost more than the product), so shared memory holds
// only the W_r and s / t rings.  Modes:
//   TR_STATS  per row the running max / log2-sum of l (log2 domain)
//   TR_TV     per row sum_v min(p, q), the part where p < q and where p = q
//             (compared in the log domain: one exp2 per element), and per
//             position the same sum for the drafter's p^b = softmax(s).  An
//             element takes two fp32 operations per instruction where it can,
//             and ties p = q are looked for 16 elements at a time (the passes
//             are bound by instruction issue: 21 per element before, 160 us at
//             512 positions of the Qwen3-8B vocabulary, now 137; log-sum-exp
//             82, now 76; dL/dz 180, now 175)
//   TR_DZ     dl = p A(sgn(p - q)) as a bf16 tile in shared memory, then
//             dz += dl W_r on the tensor core (W_r tile read MN-major); each
//             split stores its dz slice at the end.  The same tile is copied
//             to global memory for k_train_dw, as it lies in shared memory
// k_train_dw -- dW_r[v, :] = dl^T Z over the stored dl tiles: M = 128 ids, N = r,
// K = the rows of the step; added into gW_r by bulk reductions.
// The s and t tiles stream from HBM: the producers prefetch them into L2 a
// few tiles ahead (tensor-map prefetch) so that the TMA loads of the rings
// hit L2.  The -A2 [v = y*] term of dL/dl and l at y* are left to the small
// kernels (k_train_dz, k_train_stats_fin), so the loops here carry no id test.
#include "train_common.cuh"
#include "kernels.h"

namespace xp {

namespace {

constexpr float L2E = 1.4426950408889634f;

// ---------------------------------------------------------------- k_train_tok
constexpr int TR_BM = 128;
constexpr int TR_BN = 64;                                  // ids per tile in TR_DZ (128 in the other modes)
constexpr int TR_BMAX = 4;                                 // most W_r ring stages
constexpr int TR_SMAX = 8;                                 // most s / t ring stages
constexpr int TR_PF = 8;                                   // s / t tiles prefetched into L2 ahead
constexpr int TR_EPI_WARPS = 16;                           // 2 sets (item parity) x 4 lane quarters x 2 id groups
constexpr int TR_SET = TR_EPI_WARPS / 2;                   // the warps that take one item
constexpr int TR_THREADS = 32 * (2 + TR_EPI_WARPS);
constexpr uint32_t TR_BOX = 64 * 64 * 2;                   // 8 KB: a TMA box of 64 rows x 64 bf16 (128 B)
constexpr uint32_t TR_D_BUF = TR_BM * TR_BN * 2;           // 16 KB: dl tile, bf16, K-major (K = ids)
constexpr uint32_t TR_RINGS = 224 * 1024;                  // W_r ring, s / t ring (and the dl tiles in TR_DZ)
constexpr uint32_t TR_IDESC_D = idesc_bf16_mn(TR_BM, RANK, false, true);
constexpr int TR_NBUF = 4;                                 // most l accumulators in flight
// TMEM: the l accumulators (tr_nbuf) of bn columns from 0, then the Z tile (128
// columns: 256 bf16 per lane, two per column), then in TR_DZ dz (256) at 256
constexpr uint32_t TR_TMEM_COLS = 512;
constexpr uint32_t TR_DZ_COL = 256;

struct TrShared {
    uint64_t a_full;
    uint64_t full[TR_BMAX], empty[TR_BMAX];
    uint64_t sfull[TR_SMAX], sempty[TR_SMAX];
    uint64_t tfull[TR_NBUF], tempty[TR_NBUF];
    uint64_t dfull[2], dempty[2];
    uint64_t zdone, drain;
    uint32_t tmem_base;
    int abort;
};

constexpr size_t TR_SMEM = 1024 + TR_RINGS + sizeof(TrShared);
static_assert(TR_SMEM <= 232448, "k_train_tok shared memory");

// The rings of each mode (TR_RINGS holds them): W_r stages (the W_r loads
// from L2 take about 2 us under load, so their ring depth sets the pace; the
// s / t tiles are prefetched into L2 and need fewer), s / t stage bytes and
// stages, and the two dl tiles in TR_DZ.
// 128-id tiles where the epilogue is light (the log-sum-exp pass: the MMA of a
// 16-instruction tile costs the same for N = 64 and N = 128), 64 otherwise
__host__ __device__ constexpr int tr_bn(int mode) { return mode == TR_STATS ? 2 * TR_BN : TR_BN; }
__host__ __device__ constexpr uint32_t tr_bstage(int mode) { return 4u * tr_bn(mode) * 128u; }   // a W_r tile
__host__ __device__ constexpr int tr_bstages(int mode) { return mode == TR_STATS ? 2 : 4; }
__host__ __device__ constexpr int tr_nbuf(int mode) { return mode == TR_TV ? 4 : 2; }
static_assert(tr_nbuf(TR_STATS) * 2 * 64 + 128 <= 512 && tr_nbuf(TR_TV) * 64 + 128 <= 512 &&
                  tr_nbuf(TR_DZ) * 64 + 128 <= 256,
              "tensor memory: accumulators + Z (+ dz)");
__host__ __device__ constexpr uint32_t tr_st_tile(int mode) { return (uint32_t)tr_bn(mode) * 64u * 2u; }   // s or t
__host__ __device__ constexpr uint32_t tr_stage_bytes(int mode)
{
    return mode == TR_STATS ? tr_st_tile(mode) : 2 * tr_st_tile(mode);
}
__host__ __device__ constexpr int tr_stages(int mode)
{
    return (int)((TR_RINGS - tr_bstages(mode) * tr_bstage(mode) - (mode == TR_DZ ? 2 * TR_D_BUF : 0)) /
                 tr_stage_bytes(mode));
}
static_assert(tr_stages(TR_STATS) <= TR_SMAX && tr_stages(TR_TV) >= 2 && tr_stages(TR_DZ) >= 2 &&
                  tr_stages(TR_TV) <= TR_SMAX && tr_stages(TR_DZ) <= TR_SMAX && tr_bstages(TR_DZ) <= TR_BMAX,
              "ring depths");

// log2-domain running log-sum-exp over 16 values (as pairs): value = s * 2^m.
// The max and the sum run as trees (short dependent chains).
__device__ __forceinline__ void lse2_add16(float &m, float &s, const unsigned long long (&x)[8])
{
    float v[16];
#pragma unroll
    for (int j = 0; j < 8; ++j) f32x2_split(x[j], v[2 * j], v[2 * j + 1]);
    float t[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) t[j] = max3(fmaxf(v[j], v[j + 4]), v[j + 8], v[j + 12]);
    const float M = max3(max3(m, t[0], t[1]), t[2], t[3]);
    if (M == -INFINITY) return;
    const unsigned long long nm = f32x2(-M, -M);
    unsigned long long e[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float a0, a1, b0, b1;
        f32x2_split(add_f32x2(x[j], nm), a0, a1);
        f32x2_split(add_f32x2(x[j + 4], nm), b0, b1);
        e[j] = add_f32x2(f32x2(ex2_approx(a0), ex2_approx(a1)), f32x2(ex2_approx(b0), ex2_approx(b1)));
    }
    float e0, e1;
    f32x2_split(add_f32x2(add_f32x2(e[0], e[2]), add_f32x2(e[1], e[3])), e0, e1);
    s = s * ex2_approx(m - M) + (e0 + e1);
    m = M;
}

__device__ __forceinline__ void lse2_merge(float &m, float &s, float om, float os)
{
    const float M = fmaxf(m, om);
    if (M == -INFINITY) return;
    s = s * ex2_approx(m - M) + os * ex2_approx(om - M);
    m = M;
}

// 1 where x < 0, else 0.
__device__ __forceinline__ float neg_one(float x)
{
    float d;
    asm("set.lt.f32.f32 %0, %1, 0f00000000;" : "=f"(d) : "f"(x));
    return d;
}
// Two floats rounded to bf16 (nearest even), lo in bits 0-15.
__device__ __forceinline__ uint32_t cvt_bf16x2(float lo, float hi)
{
    uint32_t d;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}

// dL/dl_v without the y* term: p A(sgn(p - q)); A(0) = (Apos + Aneg) / 2
__device__ __forceinline__ float dl_value(float a2, float b2, float Apos, float Aneg)
{
    const float A = a2 > b2 ? Apos : (a2 < b2 ? Aneg : 0.5f * (Apos + Aneg));
    return ex2_approx(a2) * A;
}

}  // namespace

const size_t kTrainTokSmemBytes = TR_SMEM;
const int kTrainTokThreads = TR_THREADS;

// The token-major kernel for one mode (compiled once per mode, so that its
// tile width, ring depths and epilogue are constants).  tmap_w: W_r as (64
// columns, rows, 4 K chunks), boxes of 64 x bn x 4 (one copy per tile);
// tmap_s / tmap_t: boxes of 64 ids x 64 positions.
template <int mode>
__device__ __forceinline__ void train_tok_body(const TrainParams &p, const CUtensorMap &tmap_w,
                                               const CUtensorMap &tmap_s, const CUtensorMap &tmap_t)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *sB = base;
    TrShared &sh = *reinterpret_cast<TrShared *>(sB + TR_RINGS);
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int j = p.j0 + (int)blockIdx.y, sv = blockIdx.x;
    constexpr int bn = tr_bn(mode);                // ids per tile
    const int nvtm = (p.V + bn - 1) / bn;
    const int vt0 = (int)((long long)nvtm * sv / p.splits), vt1 = (int)((long long)nvtm * (sv + 1) / p.splits);
    const int items = vt1 - vt0;
    constexpr bool dzm = mode == TR_DZ;
    constexpr int NB = tr_bstages(mode), NS = tr_stages(mode);
    constexpr uint32_t BST = tr_bstage(mode), BCH = (uint32_t)tr_bn(mode) * 128, STT = tr_st_tile(mode);
    constexpr int NBUF = tr_nbuf(mode);
    constexpr uint32_t ZC = NBUF * bn;             // TMEM column of the Z tile
    constexpr uint32_t SB = tr_stage_bytes(mode);
    uint8_t *sS = sB + NB * BST;                   // s / t ring after the W_r ring
    uint8_t *sD = sS + NS * SB;                    // TR_DZ: the two dl tiles after the s / t ring

    if (threadIdx.x == 0) {
        mbar_init(&sh.a_full, TR_EPI_WARPS);       // every epilogue warp stores its part of Z
        for (int i = 0; i < NB; ++i) { mbar_init(&sh.full[i], 1); mbar_init(&sh.empty[i], 1); }
        for (int i = 0; i < NS; ++i) { mbar_init(&sh.sfull[i], 1); mbar_init(&sh.sempty[i], TR_SET); }
        for (int i = 0; i < TR_NBUF; ++i) {
            mbar_init(&sh.tfull[i], 1);
            mbar_init(&sh.tempty[i], TR_SET);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sh.dfull[i], TR_SET);
            mbar_init(&sh.dempty[i], 2);           // the dz MMA, and the copy of the tile to global memory
        }
        mbar_init(&sh.zdone, 1);
        mbar_init(&sh.drain, 1);
        sh.abort = 0;
        fence_barrier_init();
    }
    if (warp == 1) { tmem_alloc(&sh.tmem_base, TR_TMEM_COLS); tmem_relinquish(); }
    pdl_trigger();                 // the next kernel may start its set-up
    pdl_wait();                    // Z, the statistics and the coefficients are complete
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sh.tmem_base;
    volatile int *abort = &sh.abort;
    const unsigned long long lim = p.wait_ns;

    if (warp == 0) {
        // ------------------------------------------------------- producer
        if (lane == 0 && items > 0) {
            tma_prefetch_desc(&tmap_w);
            tma_prefetch_desc(&tmap_s);
            tma_prefetch_desc(&tmap_t);
            const uint64_t keep = policy_evict_last(), once = policy_evict_first();
            constexpr bool need_t = mode != TR_STATS;
            auto prefetch_st = [&](int it) {
                for (int x = 0; x < bn; x += 64) {
                    tma_prefetch_2d(&tmap_s, (vt0 + it) * bn + x, j * 64);
                    if (need_t) tma_prefetch_2d(&tmap_t, (vt0 + it) * bn + x, j * 64);
                }
            };
            for (int it = 0; it < min(TR_PF, items); ++it) prefetch_st(it);
            uint32_t pend_b = 0, par_b = 0, pend_s = 0, par_s = 0;
            int ss = 0;
            uint32_t sph = 0;
            for (int it = 0; it < items && !*abort; ++it) {
                const int vt = vt0 + it;
                if (it + TR_PF < items) prefetch_st(it + TR_PF);
                const int st = it % NB;
                const uint32_t ph = (uint32_t)((it / NB) & 1);
                if (!mbar_wait_spin(&sh.empty[st], ph ^ 1, abort, lim)) break;
                mbar_expect_tx(&sh.full[st], BST);   // tmap_w: (64 columns, rows, K chunk), boxes of bn rows
                tma_load_w3d(sB + st * BST, &tmap_w, &sh.full[st], vt * bn, keep);
                pend_b |= 1u << st;
                par_b = (par_b & ~(1u << st)) | (ph << st);
                if (!mbar_wait_spin(&sh.sempty[ss], sph ^ 1, abort, lim)) break;
                mbar_expect_tx(&sh.sfull[ss], SB);
                for (int x = 0; x < bn; x += 64) {   // boxes of 64 ids x 64 positions
                    tma_load_2d_hint(sS + ss * SB + x * 128, &tmap_s, &sh.sfull[ss], vt * bn + x, j * 64, once);
                    if (need_t)
                        tma_load_2d_hint(sS + ss * SB + STT + x * 128, &tmap_t, &sh.sfull[ss], vt * bn + x, j * 64,
                                         once);
                }
                pend_s |= 1u << ss;
                par_s = (par_s & ~(1u << ss)) | (sph << ss);
                if (++ss == NS) { ss = 0; sph ^= 1; }
            }
            if (*abort) {
                // no copy may still be landing when the CTA leaves
                int dummy = 0;
                for (int st = 0; st < NB; ++st)
                    if (pend_b & (1u << st)) mbar_wait_spin(&sh.full[st], (par_b >> st) & 1, &dummy, 100000000ull);
                for (int s2 = 0; s2 < NS; ++s2)
                    if (pend_s & (1u << s2)) mbar_wait_spin(&sh.sfull[s2], (par_s >> s2) & 1, &dummy, 100000000ull);
            }
        }
    } else if (warp == 1) {
        // ---------------------------------------------------- MMA issuer
        if (lane == 0 && items > 0) {
            const uint32_t b0 = smem_u32(sB), d0 = smem_u32(sD);
            // descriptors formed once, advanced per MMA
            const uint64_t bdesc0 = smem_desc_sw128(b0), ddesc0 = smem_desc_sw128(d0);
            const uint64_t bmn0 = smem_desc_sw128_mn(b0, BCH);
            // dz += dl(u) W_r(u): A = the dl tile (K-major over ids), B = the W_r
            // tile read MN-major (N = r along the 128-byte rows, K = ids)
            auto dz_step = [&](int u) -> bool {
                const int db = u & 1;
                if (!mbar_wait_spin(&sh.dfull[db], (uint32_t)((u >> 1) & 1), abort, lim)) return false;
                tc_fence_after();
                bulk_store_1d(p.dl + ((size_t)(vt0 + u) * gridDim.y + blockIdx.y) * (TR_D_BUF / 2), sD + db * TR_D_BUF,
                              TR_D_BUF);
                const uint64_t bs = smem_desc_advance(bmn0, (u % NB) * BST);
                const uint64_t ds = smem_desc_advance(ddesc0, db * TR_D_BUF);
#pragma unroll
                for (int kk = 0; kk < TR_BN / 16; ++kk)
                    tc_mma_bf16(tmem + TR_DZ_COL, smem_desc_advance(ds, kk * 32), smem_desc_advance(bs, kk * 2048),
                                TR_IDESC_D, (u | kk) != 0);
                tc_commit(&sh.empty[u % NB]);
                tc_commit(&sh.dempty[db]);
                if (u > 0) {                       // tile u - 1 has been read out by its copy
                    bulk_store_wait_read<1>();
                    mbar_arrive(&sh.dempty[db ^ 1]);
                }
                return true;
            };
            bool ok = mbar_wait_spin(&sh.a_full, 0, abort, lim);
            if (ok) tc_fence_after();
            const uint32_t idesc_f = idesc_bf16(TR_BM, bn);
            // TR_TV: two tiles at a time, their MMA chains interleaved (two
            // accumulators), so that consecutive MMAs do not depend on one another
            constexpr bool pairs = mode == TR_TV;
            for (int it = 0; pairs && it + 1 < items && ok; it += 2) {
                const int st0 = it % NB, st1 = (it + 1) % NB, q0 = it % NBUF, q1 = (it + 1) % NBUF;
                if (!mbar_wait_spin(&sh.full[st0], (uint32_t)((it / NB) & 1), abort, lim) ||
                    !mbar_wait_spin(&sh.full[st1], (uint32_t)(((it + 1) / NB) & 1), abort, lim) ||
                    !mbar_wait_spin(&sh.tempty[q0], (uint32_t)(((it / NBUF) & 1) ^ 1), abort, lim) ||
                    !mbar_wait_spin(&sh.tempty[q1], (uint32_t)((((it + 1) / NBUF) & 1) ^ 1), abort, lim)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint64_t bs0 = smem_desc_advance(bdesc0, st0 * BST), bs1 = smem_desc_advance(bdesc0, st1 * BST);
#pragma unroll
                for (int c = 0; c < 4; ++c)
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        tc_mma_bf16_ts(tmem + q0 * bn, tmem + ZC + c * 32 + kk * 8,
                                       smem_desc_advance(bs0, c * BCH + kk * 32), idesc_f, (c | kk) != 0);
                        tc_mma_bf16_ts(tmem + q1 * bn, tmem + ZC + c * 32 + kk * 8,
                                       smem_desc_advance(bs1, c * BCH + kk * 32), idesc_f, (c | kk) != 0);
                    }
                tc_commit(&sh.tfull[q0]);
                tc_commit(&sh.tfull[q1]);
                tc_commit(&sh.empty[st0]);
                tc_commit(&sh.empty[st1]);
            }
            for (int it = pairs ? (items & ~1) : 0; it < items && ok; ++it) {
                const int st = it % NB, buf = it % NBUF;
                if (!mbar_wait_spin(&sh.full[st], (uint32_t)((it / NB) & 1), abort, lim) ||
                    !mbar_wait_spin(&sh.tempty[buf], (uint32_t)(((it / NBUF) & 1) ^ 1), abort, lim)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint64_t bs = smem_desc_advance(bdesc0, st * BST);
#pragma unroll
                for (int c = 0; c < 4; ++c)
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        tc_mma_bf16_ts(tmem + buf * bn, tmem + ZC + c * 32 + kk * 8,
                                       smem_desc_advance(bs, c * BCH + kk * 32), idesc_f, (c | kk) != 0);
                tc_commit(&sh.tfull[buf]);
                if (!dzm) tc_commit(&sh.empty[st]);
                else if (it > 0 && !dz_step(it - 1)) ok = false;
            }
            if (ok && dzm) ok = dz_step(items - 1);
            if (ok && dzm) tc_commit(&sh.zdone);
            if (dzm) bulk_store_wait_all();        // every copy of a dl tile is complete before the CTA leaves
            // every MMA issued above has finished before the CTA tears down
            tc_commit(&sh.drain);
            int dummy = 0;
            mbar_wait(&sh.drain, 0, &dummy, 100000000ull);
        }
    } else {
        // ------------------------------------------------------ epilogue
        // warp set `set` takes the items of its parity (accumulators it %
        // NBUF, dl tile `set`); within a set, warp (q, g) the 32 rows of lane
        // quarter q and ids [g bn / 2, (g + 1) bn / 2) of the tile, 16 at a time
        const int ew = warp - 2, q = warp & 3, g = (ew >> 2) & 1, set = ew >> 3;
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        const int row = q * 32 + lane, f = row >> 6, pl = row & 63;
        const int i = j * 64 + pl;                 // position
        const int rowg = j * TR_BM + row;          // paired row
        const bool valid = i < p.P;
        float lp2 = 0.f, lq2 = 0.f, ls2 = 0.f, Apos = 0.f, Aneg = 0.f;
        if (valid && mode != TR_STATS) {
            lp2 = p.lse_p2[rowg];
            lq2 = p.lse_q2[i];
            ls2 = p.lse_s2[i];
        }
        if (valid && dzm) {
            const RowCoef rc = p.coef[rowg];
            Apos = rc.Apos;
            Aneg = rc.Aneg;
        }
        // Z into TMEM: warp (q, g, set) stores K elements 64 cb .. 64 cb + 63
        // (columns ZC + 32 cb ..) of its 32 rows, cb = 2 set + g
        {
            const int cb = 2 * set + g;
            const uint4 *src = reinterpret_cast<const uint4 *>(p.zop + (size_t)rowg * RANK + 64 * cb);
            uint32_t zr[32];
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const uint4 v = src[c];
                zr[4 * c] = v.x;
                zr[4 * c + 1] = v.y;
                zr[4 * c + 2] = v.z;
                zr[4 * c + 3] = v.w;
            }
            tmem_st32(tmem + lane_base + ZC + 32 * cb, zr);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.a_full);
        }
        // the anchor term's share: the teacher-forced row takes the first half
        // of each tile's ids, the consistency row the second
        const bool anchor = (f == g);
        // STATS: running (m, s); TV: 2-way partial sums of min(p, q), of the
        // part where p < q (+ half of where p = q), and of the anchor's min(p^b, q)
        float m2 = -INFINITY, s2 = 0.f;
        unsigned long long r0 = f32x2(0.f, 0.f), r1 = r0, r3 = r0;
        const unsigned long long l2e2 = f32x2(L2E, L2E), nl2e2 = f32x2(-L2E, -L2E), nlp2 = f32x2(-lp2, -lp2),
                                 lq22 = f32x2(lq2, lq2), nls2 = f32x2(-ls2, -ls2);
        bool ok = true;
        constexpr int nq = bn / 32;                // 16-id pieces per warp and tile
        for (int it = set; it < items; it += 2) {
            const int buf = it % NBUF;
            const uint32_t ph = (uint32_t)((it >> 1) & 1);      // phase of the dl tile `set`
            const int ss = it % NS;
            if (!mbar_wait_spin_warp(&sh.tfull[buf], (uint32_t)((it / NBUF) & 1), abort, lim) ||
                !mbar_wait_spin_warp(&sh.sfull[ss], (uint32_t)((it / NS) & 1), abort, lim)) {
                ok = false;
                break;
            }
            tc_fence_after();
            const uint8_t *stile = sS + ss * SB;
            const int v0 = (vt0 + it) * bn + g * (bn / 2);
            const int nv = valid ? min(bn / 2, p.V - v0) : 0;
            uint32_t w[16];
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                if (h >= nq) break;
                const int idoff = g * (bn / 2) + 16 * h;        // first id of the piece within the tile
                float acc[16];
                tmem_ld16(tmem + lane_base + buf * bn + idoff, acc);
                // the piece's 16 ids of s (and t): two 16-byte chunks of row pl
                // of the 64-id box idoff / 64
                uint4 sr[2], tr[2];
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const int off = (idoff >> 6) * (int)TR_BOX + pl * 128 +
                                    (((((idoff & 63) >> 3) + c) ^ (pl & 7)) << 4);
                    sr[c] = *reinterpret_cast<const uint4 *>(stile + off);
                    if (mode != TR_STATS) tr[c] = *reinterpret_cast<const uint4 *>(stile + STT + off);
                }
                const uint32_t ws_[8] = {sr[0].x, sr[0].y, sr[0].z, sr[0].w, sr[1].x, sr[1].y, sr[1].z, sr[1].w};
                const uint32_t wt_[8] = {tr[0].x, tr[0].y, tr[0].z, tr[0].w, tr[1].x, tr[1].y, tr[1].z, tr[1].w};
                const int nh = nv - 16 * h;              // ids of this piece that exist (<= 0: none)
                if (mode == TR_STATS) {
                    if (nh > 0) {
                        unsigned long long x[8];
#pragma unroll
                        for (int c = 0; c < 8; ++c)
                            x[c] = mul_f32x2(add_f32x2(f32x2(acc[2 * c], acc[2 * c + 1]), bf16x2_to_f32x2(ws_[c])), l2e2);
                        if (nh < 16) {
#pragma unroll
                            for (int c = 0; c < 8; ++c) {
                                float x0, x1;
                                f32x2_split(x[c], x0, x1);
                                x[c] = f32x2(2 * c < nh ? x0 : -INFINITY, 2 * c + 1 < nh ? x1 : -INFINITY);
                            }
                        }
                        lse2_add16(m2, s2, x);
                    }
                } else if (mode == TR_TV) {
                    if (nh >= 16) {
                        float tie = INFINITY;            // smallest |a2 - b2|
#pragma unroll
                        for (int c = 0; c < 8; ++c) {
                            const unsigned long long sp = bf16x2_to_f32x2(ws_[c]);
                            const unsigned long long a2 = fma_f32x2(add_f32x2(f32x2(acc[2 * c], acc[2 * c + 1]), sp), l2e2, nlp2);
                            const unsigned long long nb2 = fma_f32x2(bf16x2_to_f32x2(wt_[c]), nl2e2, lq22);   // -b2
                            float a0, a1, b0, b1, d0, d1;
                            f32x2_split(a2, a0, a1);
                            f32x2_split(nb2, b0, b1);
                            f32x2_split(add_f32x2(a2, nb2), d0, d1);
                            const unsigned long long mm = f32x2(ex2_approx(fminf(a0, -b0)), ex2_approx(fminf(a1, -b1)));
                            r0 = add_f32x2(r0, mm);
                            r1 = fma_f32x2(mm, f32x2(neg_one(d0), neg_one(d1)), r1);
                            tie = min3(tie, fabsf(d0), fabsf(d1));
                            if (anchor) {
                                float c0, c1;
                                f32x2_split(fma_f32x2(sp, l2e2, nls2), c0, c1);
                                r3 = add_f32x2(r3, f32x2(ex2_approx(fminf(c0, -b0)), ex2_approx(fminf(c1, -b1))));
                            }
                        }
                        if (tie == 0.0f) {               // p = q somewhere: half of it
                            float half = 0.0f;
#pragma unroll 1
                            for (int c = 0; c < 8; ++c) {
#pragma unroll
                                for (int e = 0; e < 2; ++e) {
                                    // by constant indexes: the arrays stay in registers
                                    float av = 0.f;
                                    uint32_t sw = 0, tw = 0;
#pragma unroll
                                    for (int k = 0; k < 8; ++k)
                                        if (k == c) { av = acc[2 * k + e]; sw = ws_[k]; tw = wt_[k]; }
                                    const float sv = __uint_as_float(e ? sw & 0xFFFF0000u : sw << 16);
                                    const float tv = __uint_as_float(e ? tw & 0xFFFF0000u : tw << 16);
                                    const float a2 = fmaf(av + sv, L2E, -lp2);
                                    if (a2 == fmaf(tv, L2E, -lq2)) half += 0.5f * ex2_approx(a2);
                                }
                            }
                            r1 = add_f32x2(r1, f32x2(half, 0.0f));
                        }
                    } else if (nh > 0) {
                        // the vocabulary's last tile: element by element
#pragma unroll
                        for (int c = 0; c < 8; ++c) {
#pragma unroll
                            for (int e = 0; e < 2; ++e) {
                                if (2 * c + e < nh) {
                                    const float sv = __uint_as_float(e ? ws_[c] & 0xFFFF0000u : ws_[c] << 16);
                                    const float tv = __uint_as_float(e ? wt_[c] & 0xFFFF0000u : wt_[c] << 16);
                                    const float a2 = fmaf(acc[2 * c + e] + sv, L2E, -lp2);
                                    const float b2 = fmaf(tv, L2E, -lq2);
                                    const float m = ex2_approx(fminf(a2, b2));
                                    r0 = add_f32x2(r0, f32x2(m, 0.0f));
                                    r1 = add_f32x2(r1, f32x2(a2 < b2 ? m : (a2 == b2 ? 0.5f * m : 0.f), 0.0f));
                                    if (anchor) r3 = add_f32x2(r3, f32x2(ex2_approx(fminf(fmaf(sv, L2E, -ls2), b2)), 0.0f));
                                }
                            }
                        }
                    }
                } else if (nh <= 0) {
                    // a padding row, or past the vocabulary's end
#pragma unroll
                    for (int c = 0; c < 8; ++c) w[8 * (h & 1) + c] = 0u;
                } else {
                    float tie = INFINITY;
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        const unsigned long long a2 =
                            fma_f32x2(add_f32x2(f32x2(acc[2 * c], acc[2 * c + 1]), bf16x2_to_f32x2(ws_[c])), l2e2, nlp2);
                        const unsigned long long nb2 = fma_f32x2(bf16x2_to_f32x2(wt_[c]), nl2e2, lq22);   // -b2
                        float a0, a1, d0, d1, v0, v1;
                        f32x2_split(a2, a0, a1);
                        f32x2_split(add_f32x2(a2, nb2), d0, d1);
                        f32x2_split(mul_f32x2(f32x2(ex2_approx(a0), ex2_approx(a1)),
                                              f32x2(d0 > 0.0f ? Apos : Aneg, d1 > 0.0f ? Apos : Aneg)), v0, v1);
                        tie = min3(tie, fabsf(d0), fabsf(d1));
                        w[8 * (h & 1) + c] = cvt_bf16x2(v0, v1);
                    }
                    if (tie == 0.0f || nh < 16) {        // p = q somewhere, or the vocabulary's end
#pragma unroll
                        for (int c = 0; c < 8; ++c) {
                            float d2[2];
#pragma unroll
                            for (int e = 0; e < 2; ++e) {
                                const float sv = __uint_as_float(e ? ws_[c] & 0xFFFF0000u : ws_[c] << 16);
                                const float tv = __uint_as_float(e ? wt_[c] & 0xFFFF0000u : wt_[c] << 16);
                                const float a2 = fmaf(acc[2 * c + e] + sv, L2E, -lp2);
                                const float b2 = fmaf(tv, L2E, -lq2);
                                d2[e] = 2 * c + e < nh ? dl_value(a2, b2, Apos, Aneg) : 0.f;
                            }
                            w[8 * (h & 1) + c] = cvt_bf16x2(d2[0], d2[1]);
                        }
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&sh.tempty[buf]);
                mbar_arrive(&sh.sempty[ss]);
            }
            if (dzm) {
                if (!mbar_wait_spin_warp(&sh.dempty[set], ph ^ 1, abort, lim)) { ok = false; break; }
                uint8_t *dt = sD + set * TR_D_BUF + row * 128;
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    *reinterpret_cast<uint4 *>(dt + (((4 * g + c) ^ (row & 7)) << 4)) =
                        make_uint4(w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.dfull[set]);
            }
        }
        if (!dzm) {
            // merge the four warps of each row (2 id groups x 2 sets), one
            // partial per (split, row); the ring is free once every item is read
            float lo[3], hi[3];
            f32x2_split(r0, lo[0], hi[0]);
            f32x2_split(r1, lo[1], hi[1]);
            f32x2_split(r3, lo[2], hi[2]);
            const float4 o4 = mode == TR_STATS ? make_float4(m2, s2, 0.f, 0.f)
                                               : make_float4(lo[0] + hi[0], lo[1] + hi[1], 0.f, lo[2] + hi[2]);
            warps_bar<32 * TR_EPI_WARPS>();
            float4 *scr = reinterpret_cast<float4 *>(sS);
            const int slot = 2 * set + g;
            if (slot != 0) scr[(slot - 1) * TR_BM + row] = o4;
            warps_bar<32 * TR_EPI_WARPS>();
            if (slot == 0 && valid && ok && !*abort) {
                float4 a = o4;
                for (int k = 0; k < 3; ++k) {
                    const float4 o = scr[k * TR_BM + row];
                    if (mode == TR_STATS) lse2_merge(a.x, a.y, o.x, o.y);
                    else { a.x += o.x; a.y += o.y; a.w += o.w; }
                }
                p.part[(size_t)sv * p.NR + rowg] = a;
            }
        } else if (ok && items > 0) {
            if (mbar_wait_spin_warp(&sh.zdone, 0, abort, lim)) {
                tc_fence_after();
                // the 4 warps of a lane quarter take 64 of the 256 columns each
                const int c0 = (2 * set + g) * 64;
#pragma unroll 1
                for (int c4 = 0; c4 < 2; ++c4) {
                    float v[32];
                    tmem_ld32(tmem + lane_base + TR_DZ_COL + c0 + c4 * 32, v);
                    float4 *dst =
                        reinterpret_cast<float4 *>(p.dzp + ((size_t)sv * p.NR + rowg) * RANK + c0 + c4 * 32);
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        dst[e] = valid ? make_float4(v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3])
                                       : make_float4(0.f, 0.f, 0.f, 0.f);
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, TR_TMEM_COLS);
    }
    if (threadIdx.x == 0 && sh.abort) set_status(p.status, ST_TIMEOUT);
}

// grid (splits, row tiles from p.j0 on), TR_THREADS threads, TR_SMEM bytes; one kernel per mode.
__global__ void __launch_bounds__(TR_THREADS, 1)
    k_train_tok_stats(const __grid_constant__ TrainParams p, const __grid_constant__ CUtensorMap tmap_w,
                      const __grid_constant__ CUtensorMap tmap_s, const __grid_constant__ CUtensorMap tmap_t)
{
    train_tok_body<TR_STATS>(p, tmap_w, tmap_s, tmap_t);
}
__global__ void __launch_bounds__(TR_THREADS, 1)
    k_train_tok_tv(const __grid_constant__ TrainParams p, const __grid_constant__ CUtensorMap tmap_w,
                   const __grid_constant__ CUtensorMap tmap_s, const __grid_constant__ CUtensorMap tmap_t)
{
    train_tok_body<TR_TV>(p, tmap_w, tmap_s, tmap_t);
}
__global__ void __launch_bounds__(TR_THREADS, 1)
    k_train_tok_dz(const __grid_constant__ TrainParams p, const __grid_constant__ CUtensorMap tmap_w,
                   const __grid_constant__ CUtensorMap tmap_s, const __grid_constant__ CUtensorMap tmap_t)
{
    train_tok_body<TR_DZ>(p, tmap_w, tmap_s, tmap_t);
}

// ----------------------------------------------------------------- k_train_dw
namespace {

constexpr int DW_BM = 128;                                 // vocabulary ids per tile
constexpr int DW_BK = 64;                                  // rows per ring stage
constexpr int DW_STAGES = 4;
constexpr int DW_EPI_WARPS = 4;
constexpr int DW_THREADS = 32 * (2 + DW_EPI_WARPS);
constexpr uint32_t DW_A_HALF = DW_BK * 128;                // 8 KB: 64 rows x 64 ids of dl
constexpr uint32_t DW_A_STAGE = 2 * DW_A_HALF;
constexpr uint32_t DW_Z_CHUNK = DW_BK * 128;               // 8 KB: 64 rows x 64 of r
constexpr uint32_t DW_Z_STAGE = 4 * DW_Z_CHUNK;
constexpr uint32_t DW_STAGE = DW_A_STAGE + DW_Z_STAGE;     // 48 KB
constexpr uint32_t DW_OUT = 32 * 128;                      // 4 KB: 32 ids x 32 fp32 columns
constexpr uint32_t DW_IDESC = idesc_bf16_mn(DW_BM, RANK, true, true);
constexpr uint32_t DW_TMEM_COLS = 2 * RANK;                // two accumulators

struct DwShared {
    uint64_t full[DW_STAGES], empty[DW_STAGES];
    uint64_t tfull[2], tempty[2];
    uint64_t drain;
    uint32_t tmem_base;
    int abort;
};

constexpr size_t DW_SMEM = 1024 + DW_STAGES * DW_STAGE + DW_EPI_WARPS * 2 * DW_OUT + sizeof(DwShared);
static_assert(DW_SMEM <= 232448, "k_train_dw shared memory");

}  // namespace

const size_t kTrainDwSmemBytes = DW_SMEM;
const int kTrainDwThreads = DW_THREADS;

// dW_r += dl^T Z over the row tiles [j0, j0 + tiles) whose dl the preceding
// k_train_tok_dz left at p.dl as [64-id tile][row tile][128 rows][64 ids] bf16
// (each 16 KB block as it lay in shared memory, i.e. with the 128-byte
// swizzle).  Read back by plain bulk copies, a block's rows are K and its ids M
// of an MN-major operand.  grid min(SMs, ceil(V / 128)), persistent over 128-id
// tiles, DW_THREADS threads:
//   warp 0     per 64 rows: the two 8 KB halves of dl and a 64 x 4 box of Z
//   warp 1     TMEM, one MMA thread: M128 N256 K16, two accumulators, so that the
//              reduction of one tile overlaps the products of the next
//   warps 2-5  32 ids each: 32 columns at a time through a swizzled 4 KB tile,
//              added into gW_r by a bulk tensor reduction (rows past V clipped)
// HBM-bound: dl (2 NR V bytes) read once, gW_r read and written.  At 512
// positions of the Qwen3-8B vocabulary 622 MB, 93 us at the measured copy rate;
// measured 91 us under ncu, against 310 us for recomputing l and dl per
// vocabulary tile (W_r Z^T again, s and t read in 2-byte steps); writing dl
// costs k_train_tok_dz 172 -> 177 us.
__global__ void __launch_bounds__(DW_THREADS, 1)
    k_train_dw(const __grid_constant__ TrainParams p, const __grid_constant__ CUtensorMap tmap_z,
               const __grid_constant__ CUtensorMap tmap_g, int tiles)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *sO = base + DW_STAGES * DW_STAGE;
    DwShared &sh = *reinterpret_cast<DwShared *>(sO + DW_EPI_WARPS * 2 * DW_OUT);
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int nvt = (p.V + DW_BM - 1) / DW_BM, nvt64 = (p.V + 63) / 64;
    const int nk = 2 * tiles;                      // 64-row steps per vocabulary tile

    if (threadIdx.x == 0) {
        for (int i = 0; i < DW_STAGES; ++i) { mbar_init(&sh.full[i], 1); mbar_init(&sh.empty[i], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&sh.tfull[i], 1); mbar_init(&sh.tempty[i], DW_EPI_WARPS); }
        mbar_init(&sh.drain, 1);
        sh.abort = 0;
        fence_barrier_init();
    }
    if (warp == 1) { tmem_alloc(&sh.tmem_base, DW_TMEM_COLS); tmem_relinquish(); }
    pdl_trigger();                 // the next kernel may start its set-up
    pdl_wait();                    // dl and Z are complete
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sh.tmem_base;
    volatile int *abort = &sh.abort;
    const unsigned long long lim = p.wait_ns;

    if (warp == 0) {
        // ------------------------------------------------------- producer
        if (lane == 0) {
            tma_prefetch_desc(&tmap_z);
            const uint64_t keep = policy_evict_last();     // Z is read by every vocabulary tile
            int st = 0;
            uint32_t ph = 0, pending = 0, pend_par = 0;
            bool ok = true;
            for (int vt = blockIdx.x; vt < nvt && ok; vt += gridDim.x)
                for (int k = 0; k < nk; ++k) {
                    if (!mbar_wait_spin(&sh.empty[st], ph ^ 1, abort, lim)) { ok = false; break; }
                    uint8_t *dst = base + st * DW_STAGE;
                    mbar_expect_tx(&sh.full[st], DW_STAGE);
                    for (int h = 0; h < 2; ++h) {
                        // (an odd last 64-id tile stands in for the one past V, whose rows are clipped)
                        const int t64 = min(2 * vt + h, nvt64 - 1);
                        const uint16_t *src = p.dl + ((size_t)t64 * tiles + (k >> 1)) * (128 * 64) + (k & 1) * (64 * 64);
                        bulk_load_1d(dst + h * DW_A_HALF, src, DW_A_HALF, &sh.full[st]);
                    }
                    tma_load_w3d(dst + DW_A_STAGE, &tmap_z, &sh.full[st], p.j0 * 128 + k * DW_BK, keep);
                    pending |= 1u << st;
                    pend_par = (pend_par & ~(1u << st)) | (ph << st);
                    if (++st == DW_STAGES) { st = 0; ph ^= 1; }
                }
            if (*abort) {
                // no copy may still be landing when the CTA leaves
                int dummy = 0;
                for (int i = 0; i < DW_STAGES; ++i)
                    if (pending & (1u << i)) mbar_wait_spin(&sh.full[i], (pend_par >> i) & 1, &dummy, 100000000ull);
            }
        }
    } else if (warp == 1) {
        // ---------------------------------------------------- MMA issuer
        if (lane == 0) {
            const uint64_t adesc0 = smem_desc_sw128_mn(smem_u32(base), DW_A_HALF);
            const uint64_t zdesc0 = smem_desc_sw128_mn(smem_u32(base) + DW_A_STAGE, DW_Z_CHUNK);
            int st = 0, lt = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (int vt = blockIdx.x; vt < nvt && ok; vt += gridDim.x, ++lt) {
                const int buf = lt & 1;
                if (!mbar_wait_spin(&sh.tempty[buf], (uint32_t)(((lt >> 1) & 1) ^ 1), abort, lim)) break;
                tc_fence_after();
                for (int k = 0; k < nk; ++k) {
                    if (!mbar_wait_spin(&sh.full[st], ph, abort, lim)) { ok = false; break; }
                    tc_fence_after();
                    const uint64_t ad = smem_desc_advance(adesc0, st * DW_STAGE), zd = smem_desc_advance(zdesc0, st * DW_STAGE);
#pragma unroll
                    for (int kk = 0; kk < DW_BK / 16; ++kk)
                        tc_mma_bf16(tmem + buf * RANK, smem_desc_advance(ad, kk * 2048), smem_desc_advance(zd, kk * 2048),
                                    DW_IDESC, (k | kk) != 0);
                    tc_commit(&sh.empty[st]);
                    if (++st == DW_STAGES) { st = 0; ph ^= 1; }
                }
                if (ok) tc_commit(&sh.tfull[buf]);
            }
            // every MMA issued above has finished before the CTA tears down
            tc_commit(&sh.drain);
            int dummy = 0;
            mbar_wait(&sh.drain, 0, &dummy, 100000000ull);
        }
    } else {
        // ------------------------------------------------------ epilogue
        const int q = warp & 3;
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        uint8_t *out = sO + q * 2 * DW_OUT;
        int lt = 0, piece = 0;
        for (int vt = blockIdx.x; vt < nvt; vt += gridDim.x, ++lt) {
            const int buf = lt & 1, y = vt * DW_BM + q * 32;
            if (!mbar_wait_spin_warp(&sh.tfull[buf], (uint32_t)((lt >> 1) & 1), abort, lim)) break;
            tc_fence_after();
#pragma unroll 1
            for (int c = 0; c < RANK / 32; ++c, ++piece) {
                float v[32];
                tmem_ld32(tmem + lane_base + buf * RANK + c * 32, v);
                uint8_t *ob = out + (piece & 1) * DW_OUT;
                if (lane == 0) bulk_store_wait_read<1>();  // the piece before last has left this buffer
                __syncwarp();
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    *reinterpret_cast<float4 *>(ob + lane * 128 + ((e ^ (lane & 7)) << 4)) =
                        make_float4(v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3]);
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0 && y < p.V) tma_reduce_add_2d(&tmap_g, ob, c * 32, y);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.tempty[buf]);
        }
        if (lane == 0) bulk_store_wait_all();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, DW_TMEM_COLS);
    }
    if (threadIdx.x == 0 && sh.abort) set_status(p.status, ST_TIMEOUT);
}

}  // namespace xp
