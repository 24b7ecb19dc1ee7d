// train_kernels.cu -- the memory-bound and per-block steps of the refiner
// training step (Sec. 4.3) around the tensor-core products.  Every kernel of
// the step is launched with programmatic dependent launch: it signals its
// successor at once and waits for its predecessor before touching memory.
//
//   k_train_rows / _fin   one pass over s and the target logits t of every
//                         position: log-sum-exp of both (log2 domain), s at
//                         y*, and the first argmax of s (the consistency
//                         forward's inputs, argmax p^b)
//   k_train_fuse          the Fuse operand [u_h | u_g | W_e[x]] of both
//                         forwards (Eq. fuse; u_g = W_g g with g the block
//                         mean of h, taken as the mean of W_g h_j), u_h and
//                         u_g as bf16 hi + lo pairs so that W_in sees them to
//                         about 16 bits
//   k_train_mix           c_k = a_k + sum_{j<k} L_kj a_j per channel (Eq. mix),
//                         L staged in shared memory per 32 channels
//   k_train_stats_fin     lse of every row's logits from the split partials
//   k_train_tv_fin        per block the three losses and L_total; per row the
//                         coefficients of dL/dl
//   k_train_dz, _dact     dL/dz from the vocabulary splits and its bf16 copy;
//                         dL/dt = dL/du sigma'(t)
//   k_train_mix_bwd       dL/da_j = dc_j + sum_{k>j} L_kj dc_k and dL/dL_kj
//   k_train_fuse_bwd      dL/du_h per position (both forwards), dL/du_g / B
//                         per block, dL/dW_e rows (atomic, both forwards)
#include "train_common.cuh"
#include "kernels.h"

namespace xp {

namespace {

constexpr float L2E = 1.4426950408889634f;
constexpr float LN2 = 0.69314718055994531f;

__device__ __forceinline__ int pair_row(int i, int f) { return (i >> 6) * 128 + f * 64 + (i & 63); }

__device__ __forceinline__ void lse2_merge(float &m, float &s, float om, float os)
{
    const float M = fmaxf(m, om);
    if (M == -INFINITY) return;
    s = s * ex2_approx(m - M) + os * ex2_approx(om - M);
    m = M;
}

__device__ __forceinline__ float sigma_prime(int act, float t)
{
    if (act == 2) return t > 0.0f ? 1.0f : 0.0f;
    if (act == 1)
        return 0.5f * (1.0f + erff(t * 0.70710678118654752f)) + t * 0.39894228040143268f * expf(-0.5f * t * t);
    const float sg = 1.0f / (1.0f + expf(-t));
    return sg + t * sg * (1.0f - sg);
}

}  // namespace

namespace {

constexpr int ROWS_STAGES = 3;
constexpr uint32_t ROWS_SEG = TRAIN_ROW_CHUNK * 2;          // bytes of one s (or t) segment
constexpr int ROWS_THREADS = 32 * 10;                        // a copy warp, 8 reducing warps, a merging warp
constexpr int ROWS_PART = 4;                                 // items whose partials wait for the merging warp

struct RowsShared {
    uint64_t full[ROWS_STAGES], empty[ROWS_STAGES];
    uint64_t pfull[ROWS_PART], pempty[ROWS_PART];
    float4 wp[ROWS_PART][8];                                  // per item and warp: max / sum of s and t
    float wb[ROWS_PART][8];
    int wi[ROWS_PART][8];
    int abort;
};

constexpr size_t ROWS_SMEM = 128 + ROWS_STAGES * 2 * ROWS_SEG + sizeof(RowsShared);

}  // namespace

const size_t kTrainRowsSmemBytes = ROWS_SMEM;
const int kTrainRowsThreads = ROWS_THREADS;

// grid min(SMs, P nch), ROWS_THREADS threads, ROWS_SMEM bytes: persistent
// over the (position, chunk of TRAIN_ROW_CHUNK ids) items, position-major.
// Warp 0 streams each item's s and t segments into a ROWS_STAGES-deep ring by
// bulk copies; reducing warp w takes the 8-id pieces 32 w + lane + 256 c
// (c < 8), so each of its shared-memory reads is one 512-byte run, and
// releases the stage as soon as its pieces are in registers.  The warp's
// maxima are reduced first (on the packed words), so every exponential is taken
// against the warp maximum and the sums need no rescale; the id of the maximum is
// looked for by the lanes that hold it.  A last warp merges an item's 8 partials,
// so that no barrier makes the reducing warps wait for one another: with a merge
// by one thread between two barriers per item 512 positions of the Qwen3-8B
// vocabulary took 71 us, now 61 (311 MB: 47 us at the copy bandwidth).
__global__ void __launch_bounds__(ROWS_THREADS, 1) k_train_rows(TrainMisc m)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
    RowsShared &sh = *reinterpret_cast<RowsShared *>(base + ROWS_STAGES * 2 * ROWS_SEG);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int items = m.P * m.nch;
    if (threadIdx.x == 0) {
        for (int i = 0; i < ROWS_STAGES; ++i) {
            mbar_init(&sh.full[i], 1);
            mbar_init(&sh.empty[i], 8);
        }
        for (int i = 0; i < ROWS_PART; ++i) {
            mbar_init(&sh.pfull[i], 8);
            mbar_init(&sh.pempty[i], 1);
        }
        sh.abort = 0;
        fence_barrier_init();
    }
    __syncthreads();
    pdl_trigger();
    pdl_wait();
    volatile int *abort = &sh.abort;
    if (warp == 0) {
        if (lane == 0) {
            uint32_t pending = 0, pend_par = 0;
            int k = 0;
            for (int it = blockIdx.x; it < items; it += gridDim.x, ++k) {
                const int st = k % ROWS_STAGES;
                const uint32_t ph = (uint32_t)((k / ROWS_STAGES) & 1);
                if (!mbar_wait(&sh.empty[st], ph ^ 1, abort)) break;
                const int i = it / m.nch, v0 = (it % m.nch) * TRAIN_ROW_CHUNK;
                // V % 8 == 0: the segment's bytes are a multiple of 16
                const uint32_t bytes = (uint32_t)min(TRAIN_ROW_CHUNK, m.V - v0) * 2u;
                uint8_t *dst = base + st * 2 * ROWS_SEG;
                mbar_expect_tx(&sh.full[st], 2 * bytes);
                bulk_load_1d(dst, static_cast<const uint16_t *>(m.s) + (size_t)i * m.V + v0, bytes, &sh.full[st]);
                bulk_load_1d(dst + ROWS_SEG, static_cast<const uint16_t *>(m.t) + (size_t)i * m.V + v0, bytes,
                             &sh.full[st]);
                pending |= 1u << st;
                pend_par = (pend_par & ~(1u << st)) | (ph << st);
            }
            if (*abort) {
                // no copy may still be landing when the CTA leaves
                int dummy = 0;
                for (int st = 0; st < ROWS_STAGES; ++st)
                    if (pending & (1u << st)) mbar_wait(&sh.full[st], (pend_par >> st) & 1, &dummy, 100000000ull);
            }
        }
    } else if (warp <= 8) {
        const int w = warp - 1;
        constexpr uint32_t NEG2 = 0xFF80FF80u;   // two bf16 -inf
        int k = 0;
        for (int it = blockIdx.x; it < items; it += gridDim.x, ++k) {
            const int st = k % ROWS_STAGES;
            if (!mbar_wait_warp(&sh.full[st], (uint32_t)((k / ROWS_STAGES) & 1), abort)) break;
            const int ch = it % m.nch, v0 = ch * TRAIN_ROW_CHUNK, n = min(TRAIN_ROW_CHUNK, m.V - v0);
            const uint4 *ss = reinterpret_cast<const uint4 *>(base + st * 2 * ROWS_SEG);
            const uint4 *tt = ss + ROWS_SEG / 16;
            uint4 ps[8], pt[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const int pc = 32 * w + lane + 256 * c;
                if (8 * pc < n) {
                    ps[c] = ss[pc];
                    pt[c] = tt[pc];
                } else {
                    ps[c] = pt[c] = make_uint4(NEG2, NEG2, NEG2, NEG2);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.empty[st]);
            // maxima on the packed words (exact; NaN loses to any number)
            uint32_t xs[2] = {NEG2, NEG2}, xt[2] = {NEG2, NEG2};
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                xs[c & 1] = max_bf16x2(max_bf16x2(xs[c & 1], max_bf16x2(ps[c].x, ps[c].y)), max_bf16x2(ps[c].z, ps[c].w));
                xt[c & 1] = max_bf16x2(max_bf16x2(xt[c & 1], max_bf16x2(pt[c].x, pt[c].y)), max_bf16x2(pt[c].z, pt[c].w));
            }
            const uint32_t xs1 = max_bf16x2(xs[0], xs[1]), xt1 = max_bf16x2(xt[0], xt[1]);
            const float mine = fmaxf(__uint_as_float(xs1 << 16), __uint_as_float(xs1 & 0xFFFF0000u));
            float best = mine, mt = fmaxf(__uint_as_float(xt1 << 16), __uint_as_float(xt1 & 0xFFFF0000u));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, o));
                mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, o));
            }
            // best is now the warp's maximum of s (log2 domain below)
            const float ms2 = best * L2E, mt2 = mt * L2E;
            const bool has_s = best != -INFINITY, has_t = mt != -INFINITY;
            // its first id: a lane that holds it walks its ids (increasing along c,
            // word, half) backwards
            int idx = 0x7fffffff;
            if (has_s && mine == best) {
                const int vt = v0 + 8 * (32 * w + lane);
#pragma unroll
                for (int c = 7; c >= 0; --c) {
                    const uint32_t ws[4] = {ps[c].x, ps[c].y, ps[c].z, ps[c].w};
#pragma unroll
                    for (int q = 3; q >= 0; --q) {
                        if (__uint_as_float(ws[q] & 0xFFFF0000u) == best) idx = vt + 2048 * c + 2 * q + 1;
                        if (__uint_as_float(ws[q] << 16) == best) idx = vt + 2048 * c + 2 * q;
                    }
                }
            }
            __syncwarp();
            idx = __reduce_min_sync(0xffffffffu, idx);
            unsigned long long sa2[2] = {0, 0}, ta2[2] = {0, 0};      // pairs of partial sums
            const unsigned long long l2 = f32x2(L2E, L2E), ns2 = f32x2(-ms2, -ms2), nt2 = f32x2(-mt2, -mt2);
            auto add = [&](unsigned long long &sum, uint32_t word, unsigned long long nm) {
                float e0, e1;
                f32x2_split(fma_f32x2(bf16x2_to_f32x2(word), l2, nm), e0, e1);
                sum = add_f32x2(sum, f32x2(ex2_approx(e0), ex2_approx(e1)));
            };
            if (has_s)
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    add(sa2[0], ps[c].x, ns2); add(sa2[1], ps[c].y, ns2);
                    add(sa2[0], ps[c].z, ns2); add(sa2[1], ps[c].w, ns2);
                }
            if (has_t)
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    add(ta2[0], pt[c].x, nt2); add(ta2[1], pt[c].y, nt2);
                    add(ta2[0], pt[c].z, nt2); add(ta2[1], pt[c].w, nt2);
                }
            float sa[2], ta[2];
            f32x2_split(add_f32x2(sa2[0], sa2[1]), sa[0], sa[1]);
            f32x2_split(add_f32x2(ta2[0], ta2[1]), ta[0], ta[1]);
            float sum_s = sa[0] + sa[1], sum_t = ta[0] + ta[1];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                sum_s += __shfl_xor_sync(0xffffffffu, sum_s, o);
                sum_t += __shfl_xor_sync(0xffffffffu, sum_t, o);
            }
            const int pb = k % ROWS_PART;
            if (lane == 0 && mbar_wait(&sh.pempty[pb], (uint32_t)((k / ROWS_PART) & 1) ^ 1, abort)) {
                sh.wp[pb][w] = make_float4(has_s ? ms2 : -INFINITY, sum_s, has_t ? mt2 : -INFINITY, sum_t);
                sh.wb[pb][w] = best;
                sh.wi[pb][w] = idx;
                mbar_arrive(&sh.pfull[pb]);
            }
        }
    } else {
        // the merging warp: the 8 partials of an item (lanes 0-7), while the
        // reducing warps go on
        int k = 0;
        for (int it = blockIdx.x; it < items; it += gridDim.x, ++k) {
            const int pb = k % ROWS_PART;
            if (!mbar_wait_warp(&sh.pfull[pb], (uint32_t)((k / ROWS_PART) & 1), abort)) break;
            float4 a = make_float4(-INFINITY, 0.f, -INFINITY, 0.f);
            float b = -INFINITY;
            int bi = 0x7fffffff;
            if (lane < 8) {
                a = sh.wp[pb][lane];
                b = sh.wb[pb][lane];
                bi = sh.wi[pb][lane];
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.pempty[pb]);
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) {
                const float om = __shfl_xor_sync(0xffffffffu, a.x, o), os = __shfl_xor_sync(0xffffffffu, a.y, o);
                const float pm = __shfl_xor_sync(0xffffffffu, a.z, o), ps = __shfl_xor_sync(0xffffffffu, a.w, o);
                const float ob = __shfl_xor_sync(0xffffffffu, b, o);
                const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                lse2_merge(a.x, a.y, om, os);
                lse2_merge(a.z, a.w, pm, ps);
                merge_argmax(b, bi, ob, oi);
            }
            if (lane == 0) {
                m.rpart[it] = a;                 // item i nch + ch
                m.rkey[it] = argmax_key(b, bi);
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && sh.abort) set_status(m.status, ST_TIMEOUT);
}

// grid ceil(P / 8), 256 threads: one warp per position.
__global__ void __launch_bounds__(256) k_train_rows_fin(TrainMisc m)
{
    pdl_trigger();
    pdl_wait();
    const int i = blockIdx.x * 8 + threadIdx.x / 32, lane = threadIdx.x % 32;
    if (i >= m.P) return;
    float ms = -INFINITY, ss = 0.f, mt = -INFINITY, st = 0.f;
    unsigned long long key = 0;
    for (int c = lane; c < m.nch; c += 32) {
        const float4 a = m.rpart[(size_t)i * m.nch + c];
        lse2_merge(ms, ss, a.x, a.y);
        lse2_merge(mt, st, a.z, a.w);
        key = max(key, m.rkey[(size_t)i * m.nch + c]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lse2_merge(ms, ss, __shfl_xor_sync(0xffffffffu, ms, o), __shfl_xor_sync(0xffffffffu, ss, o));
        lse2_merge(mt, st, __shfl_xor_sync(0xffffffffu, mt, o), __shfl_xor_sync(0xffffffffu, st, o));
        key = max(key, __shfl_xor_sync(0xffffffffu, key, o));
    }
    if (lane == 0) {
        m.lse_s2[i] = ms + log2f(ss);
        m.lse_q2[i] = mt + log2f(st);
        int y = m.ystar[i];
        if (y < 0 || y >= m.V) {
            set_status(m.status, ST_BOUNDS);
            y = 0;
        }
        m.s_y[i] = bf2f(static_cast<const uint16_t *>(m.s)[(size_t)i * m.V + y]);
        if (m.xhat_in) {
            m.xhat[i] = m.xhat_in[i];
        } else {
            float b;
            int bi;
            argmax_unkey(key, b, bi);
            m.xhat[i] = bi;
        }
    }
}

// grid (b + ceil((NR / 2 - P) / B), r / 32), block (32, B): position y of block
// blockIdx.x (past b: a padding position, zeroed), channel 32 blockIdx.y + x.
// Latency-bound on the K-split slices of W_h h and W_g h, at most 152 of each
// per element: every (position, channel) has its own thread, which requests its
// slices together and adds them in a fixed order (with 256 threads per four
// positions walking all positions' slices in turn 24 slices took 48 us at 96
// positions and 8 slices 22 us at 512, now 7 and 6).  u_g, the mean of
// the block, meets in shared memory.
__global__ void __launch_bounds__(1024) k_train_fuse(TrainMisc m)
{
    pdl_trigger();
    pdl_wait();
    const int d = blockIdx.y * 32 + threadIdx.x, k = threadIdx.y, B = m.B, r5 = 5 * RANK;
    const int blk = blockIdx.x;
    if (blk >= m.b) {
        // padding rows: zero operands and activations so that every product
        // over them vanishes
        const int i = m.P + (blk - m.b) * B + k;
        if (i >= m.NR / 2) return;
        for (int f = 0; f < 2; ++f) {
            const int row = pair_row(i, f);
            for (int c = 0; c < 5; ++c) m.X[(size_t)row * r5 + c * RANK + d] = 0;
            m.c[(size_t)row * RANK + d] = 0.f;
            m.cop[(size_t)row * RANK + d] = 0;
            m.dab[(size_t)row * RANK + d] = 0;
            if (d == 0) m.xrow[row] = -1;
        }
        return;
    }
    __shared__ float su[MAX_B][32];
    const int i = blk * B + k;
    // the K-split slices of W_h h and W_g h, summed in a fixed order
    const size_t slice = (size_t)m.P * RANK;
    const float *ph = m.Uh + (size_t)i * RANK + d, *pg = m.Ug + (size_t)i * RANK + d;
    float uhv = 0.f, uj = 0.f;
    for (int s0 = 0; s0 < m.usplits; s0 += 8) {
        float vh[8], vg[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            vh[q] = s0 + q < m.usplits ? ph[(s0 + q) * slice] : 0.f;
            vg[q] = s0 + q < m.usplits ? pg[(s0 + q) * slice] : 0.f;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            uhv += vh[q];
            uj += vg[q];
        }
    }
    su[k][threadIdx.x] = uj;
    int x[2];
    for (int f = 0; f < 2; ++f) {
        x[f] = k == 0 ? m.anchor[blk] : (f == 0 ? m.ystar[i - 1] : m.xhat[i - 1]);
        if (x[f] < 0 || x[f] >= m.V) {
            if (d == 0) set_status(m.status, ST_BOUNDS);
            x[f] = 0;
        }
    }
    const uint16_t we[2] = {m.W_e[(size_t)x[0] * RANK + d], m.W_e[(size_t)x[1] * RANK + d]};
    __syncthreads();
    float ug = 0.f;
    for (int j = 0; j < B; ++j) ug += su[j][threadIdx.x];
    ug /= (float)B;
    const uint16_t ugb = f2bf(ug), ugl = f2bf(ug - bf2f(ugb));
    const uint16_t uh = f2bf(uhv), uhl = f2bf(uhv - bf2f(uh));
    for (int f = 0; f < 2; ++f) {
        const int row = pair_row(i, f);
        uint16_t *X = m.X + (size_t)row * r5 + d;
        X[0] = uh;
        X[RANK] = ugb;
        X[2 * RANK] = we[f];
        X[3 * RANK] = uhl;
        X[4 * RANK] = ugl;
        if (d == 0) m.xrow[row] = x[f];
    }
}

namespace {

// The causal mixer of 32 channels, staged as Ls[(k B + j) 32 + d] (fp32,
// channel innermost); only j < k is read.  From the caller's L and not the
// refiner's packed copy: a training loop may update its weights in place.
__device__ __forceinline__ void stage_L(const TrainMisc &m, float *Ls, int d0)
{
    const int B = m.B, n = 32 * B * B;
    for (int e = threadIdx.y * 32 + threadIdx.x; e < n; e += 32 * B) {
        const int dl = e / (B * B), kj = e % (B * B);
        Ls[kj * 32 + dl] = bf2f(m.L[(size_t)(d0 + dl) * B * B + kj]);
    }
}

inline size_t mix_smem(int B) { return (size_t)(32 * B * B + 2 * B * 32) * 4; }

}  // namespace

size_t train_mix_smem(int B) { return mix_smem(B); }

// grid (r / 32, ceil(2 b / mseq)), block (32, B): channel d0 + x, position y
// of the sequences 2 blk + f of the CTA's group: c_k = a_k + sum_{j<k} L_kj a_j.
__global__ void __launch_bounds__(1024) k_train_mix(TrainMisc m)
{
    pdl_trigger();
    extern __shared__ float smf[];
    const int B = m.B, dl = threadIdx.x, k = threadIdx.y, d0 = blockIdx.x * 32, d = d0 + dl;
    float *Ls = smf, *sa = smf + 32 * B * B;
    stage_L(m, Ls, d0);
    pdl_wait();
    for (int q = 0; q < m.mseq; ++q) {
        const int sq = blockIdx.y * m.mseq + q;
        if (sq >= 2 * m.b) break;
        const int blk = sq >> 1, f = sq & 1;
        const int row = pair_row(blk * B + k, f);
        const float ak = m.a[(size_t)row * RANK + d];
        __syncthreads();                           // Ls staged; the previous sequence's sa read
        sa[k * 32 + dl] = ak;
        __syncthreads();
        float acc = ak;
        for (int j = 0; j < k; ++j) acc = fmaf(Ls[(k * B + j) * 32 + dl], sa[j * 32 + dl], acc);
        m.c[(size_t)row * RANK + d] = acc;
        m.cop[(size_t)row * RANK + d] = f2bf(acc);
    }
}

// Same grid: dL/da_j = dc_j + sum_{k>j} L_kj dc_k, and this group's share of
// dL/dL_kj = sum over sequences of dc_k a_j (added atomically into gL, once per
// group: the atomics of 32 channels are 32 cache lines).
__global__ void __launch_bounds__(1024) k_train_mix_bwd(TrainMisc m)
{
    pdl_trigger();
    extern __shared__ float smf[];
    const int B = m.B, dl = threadIdx.x, j = threadIdx.y, d0 = blockIdx.x * 32, d = d0 + dl;
    float *Ls = smf, *sdc = smf + 32 * B * B, *sa = sdc + B * 32;
    stage_L(m, Ls, d0);
    pdl_wait();
    float gl[MAX_B];                               // thread (d, k = j) holds dL/dL_kj' for j' < k
    for (int jj = 0; jj < MAX_B; ++jj) gl[jj] = 0.f;
    for (int q = 0; q < m.mseq; ++q) {
        const int sq = blockIdx.y * m.mseq + q;
        if (sq >= 2 * m.b) break;
        const int blk = sq >> 1, f = sq & 1;
        const int row = pair_row(blk * B + j, f);
        const float dcj = m.dc[(size_t)row * RANK + d];
        const float aj = m.a[(size_t)row * RANK + d];
        __syncthreads();
        sdc[j * 32 + dl] = dcj;
        sa[j * 32 + dl] = aj;
        __syncthreads();
        float acc = dcj;
        for (int k = j + 1; k < B; ++k) acc = fmaf(Ls[(k * B + j) * 32 + dl], sdc[k * 32 + dl], acc);
        m.dab[(size_t)row * RANK + d] = f2bf(acc);
#pragma unroll
        for (int jj = 0; jj < MAX_B; ++jj)
            if (jj < j) gl[jj] = fmaf(dcj, sa[jj * 32 + dl], gl[jj]);
    }
#pragma unroll
    for (int jj = 0; jj < MAX_B; ++jj)
        if (jj < j) atomicAdd(m.gL + ((size_t)d * B + j) * B + jj, gl[jj]);
}

// grid NR / 8, 256 threads: one warp per row.  The row's log-sum-exp from the
// split partials, and its logit at y*: s_y* + W_r[y*] . z (the bf16 operands
// of the Read, fp32 accumulation).
__global__ void __launch_bounds__(256) k_train_stats_fin(TrainMisc m)
{
    pdl_trigger();
    pdl_wait();
    const int row = blockIdx.x * 8 + threadIdx.x / 32, lane = threadIdx.x % 32;
    if (row >= m.NR) return;
    const int i = (row >> 7) * 64 + (row & 63);
    if (i >= m.P) {
        if (lane == 0) {
            m.lse_p2[row] = 0.f;
            m.ly[row] = 0.f;
        }
        return;
    }
    float mx = -INFINITY, s = 0.f;
    for (int sv = lane; sv < m.splits; sv += 32) {
        const float4 a = m.part[(size_t)sv * m.NR + row];
        lse2_merge(mx, s, a.x, a.y);
    }
    int y = m.ystar[i];
    if (y < 0 || y >= m.V) y = 0;                 // reported by k_train_rows_fin
    // lane: 8 consecutive elements of the 256
    const uint4 a = reinterpret_cast<const uint4 *>(m.W_r + (size_t)y * RANK)[lane];
    const uint4 b = reinterpret_cast<const uint4 *>(m.zop + (size_t)row * RANK)[lane];
    const uint32_t wa[4] = {a.x, a.y, a.z, a.w}, wb[4] = {b.x, b.y, b.z, b.w};
    float acc = 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        acc = fmaf(__uint_as_float(wa[q] << 16), __uint_as_float(wb[q] << 16), acc);
        acc = fmaf(__uint_as_float(wa[q] & 0xFFFF0000u), __uint_as_float(wb[q] & 0xFFFF0000u), acc);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        acc += __shfl_xor_sync(0xffffffffu, acc, o);
        lse2_merge(mx, s, __shfl_xor_sync(0xffffffffu, mx, o), __shfl_xor_sync(0xffffffffu, s, o));
    }
    if (lane == 0) {
        m.lse_p2[row] = mx + log2f(s);
        m.ly[row] = m.s_y[i] + acc;
    }
}

// grid b, block (32, B): warp k = position k of block blockIdx.x, its lanes the
// vocabulary splits of the position's two rows (a fixed tree; one thread per
// position walking 76 splits in turn took 20 us, now 6).
__global__ void __launch_bounds__(1024) k_train_tv_fin(TrainMisc m)
{
    pdl_trigger();
    pdl_wait();
    const int blk = blockIdx.x, k = threadIdx.y, lane = threadIdx.x;
    const int i = blk * m.B + k;
    __shared__ float sl[3][MAX_B];
    float sum[2][2] = {{0.f, 0.f}, {0.f, 0.f}}, anc = 0.f;   // per forward: x, y of the partials
    for (int sv = lane; sv < m.splits; sv += 32) {
#pragma unroll
        for (int f = 0; f < 2; ++f) {
            const float4 a = m.part[(size_t)sv * m.NR + pair_row(i, f)];
            sum[f][0] += a.x;
            sum[f][1] += a.y;
            anc += a.w;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int f = 0; f < 2; ++f)
#pragma unroll
            for (int q = 0; q < 2; ++q) sum[f][q] += __shfl_xor_sync(0xffffffffu, sum[f][q], o);
        anc += __shfl_xor_sync(0xffffffffu, anc, o);
    }
    if (lane == 0) {
        const float w = expf(-(float)k / m.gamma);
        float lf[2];
        for (int f = 0; f < 2; ++f) {
            const int row = pair_row(i, f);
            const float sm = sum[f][0], lt = sum[f][1];
            // lt: sum of p where p < q plus half of it where p = q (k_train_tok)
            const float l1 = 2.0f * (1.0f - sm);
            const float S = 1.0f - 2.0f * lt;               // sum_v sgn(p_v - q_v) p_v
            const float ce = m.lse_p2[row] * LN2 - m.ly[row];
            lf[f] = w * (m.a_ce * ce + m.a_l1 * l1);
            // dL/dl_v = cf [a_ce (p_v - [v = y*]) + a_l1 p_v (sgn(p_v - q_v) - S)]
            const float cf = w * (f == 0 ? 1.0f : m.beta);
            RowCoef rc;
            rc.lse_p2 = m.lse_p2[row];
            rc.lse_q2 = m.lse_q2[i];
            rc.Apos = cf * (m.a_ce + m.a_l1 * (1.0f - S));
            rc.Aneg = cf * (m.a_ce - m.a_l1 * (1.0f + S));
            m.coef[row] = rc;
            m.A2[row] = cf * m.a_ce;
        }
        const float ceb = m.lse_s2[i] * LN2 - m.s_y[i];
        sl[0][k] = lf[0];
        sl[1][k] = w * (m.a_ce * ceb + m.a_l1 * 2.0f * (1.0f - anc));
        sl[2][k] = lf[1];
    }
    __syncthreads();
    if (k == 0) {
        float v[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) v[q] = lane < m.B ? sl[q][lane] : 0.f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int q = 0; q < 3; ++q) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
        if (lane == 0) {
            m.loss[blk * 4 + 0] = v[0];
            m.loss[blk * 4 + 1] = v[1];
            m.loss[blk * 4 + 2] = v[2];
            m.loss[blk * 4 + 3] = v[0] + m.lambda * v[1] + m.beta * v[2];
        }
    }
}

// grid ceil(NR r / 256), 256 threads, four threads per 4 elements: dL/dz as the
// sum of the vocabulary splits' slices in a fixed order (thread q of the four
// takes the splits q, q + 4, ...; 76 slices in turn took 15 us, now 10) plus the
// -A2 [v = y*] term of dL/dl (-A2 W_r[y*]), and its bf16 copy; the same term of
// dL/dW_r, -A2 z at row y*, is added into gW_r (atomic: positions share ids).
__global__ void __launch_bounds__(256) k_train_dz(TrainMisc m)
{
    pdl_trigger();
    pdl_wait();
    const size_t e = (((size_t)blockIdx.x * 256 + threadIdx.x) >> 2) * 4;   // NR r is a multiple of 256
    const size_t n = (size_t)m.NR * RANK;
    const int q = threadIdx.x & 3;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 5
    for (int sp = q; sp < m.splits; sp += 4) {
        const float4 o = *reinterpret_cast<const float4 *>(m.dzp + sp * n + e);
        v.x += o.x;
        v.y += o.y;
        v.z += o.z;
        v.w += o.w;
    }
#pragma unroll
    for (int o = 1; o <= 2; o <<= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
        v.z += __shfl_xor_sync(0xffffffffu, v.z, o);
        v.w += __shfl_xor_sync(0xffffffffu, v.w, o);
    }
    if (q != 0) return;
    const int row = (int)(e / RANK), d = (int)(e % RANK);
    const float a2 = m.A2[row];
    if (a2 != 0.0f) {
        int y = m.ystar[(row >> 7) * 64 + (row & 63)];
        if (y < 0 || y >= m.V) y = 0;             // reported by k_train_rows_fin
        const uint2 wv = *reinterpret_cast<const uint2 *>(m.W_r + (size_t)y * RANK + d);
        v.x -= a2 * __uint_as_float(wv.x << 16);
        v.y -= a2 * __uint_as_float(wv.x & 0xFFFF0000u);
        v.z -= a2 * __uint_as_float(wv.y << 16);
        v.w -= a2 * __uint_as_float(wv.y & 0xFFFF0000u);
        const uint2 zv = *reinterpret_cast<const uint2 *>(m.zop + (size_t)row * RANK + d);
        float *g = m.gW_r + (size_t)y * RANK + d;
        atomicAdd(g + 0, -a2 * __uint_as_float(zv.x << 16));
        atomicAdd(g + 1, -a2 * __uint_as_float(zv.x & 0xFFFF0000u));
        atomicAdd(g + 2, -a2 * __uint_as_float(zv.y << 16));
        atomicAdd(g + 3, -a2 * __uint_as_float(zv.y & 0xFFFF0000u));
    }
    *reinterpret_cast<float4 *>(m.dz + e) = v;
    *reinterpret_cast<uint2 *>(m.dzb + e) = make_uint2(pack_bf16x2(v.x, v.y), pack_bf16x2(v.z, v.w));
}

// grid ceil(NR 2r / 1024), 256 threads: dL/dt = dL/du sigma'(t), 4 elements each.
__global__ void __launch_bounds__(256) k_train_dact(TrainMisc m)
{
    pdl_trigger();
    pdl_wait();
    const size_t e = ((size_t)blockIdx.x * 256 + threadIdx.x) * 4;
    if (e >= (size_t)m.NR * 2 * RANK) return;
    const float4 du = *reinterpret_cast<const float4 *>(m.du + e);
    const float4 t = *reinterpret_cast<const float4 *>(m.tpre + e);
    *reinterpret_cast<uint2 *>(m.dtb + e) =
        make_uint2(pack_bf16x2(du.x * sigma_prime(m.act, t.x), du.y * sigma_prime(m.act, t.y)),
                   pack_bf16x2(du.z * sigma_prime(m.act, t.z), du.w * sigma_prime(m.act, t.w)));
}

// grid P, r threads.
__global__ void __launch_bounds__(RANK) k_train_fuse_bwd(TrainMisc m)
{
    pdl_trigger();
    pdl_wait();
    const int i = blockIdx.x, d = threadIdx.x, r3 = 3 * RANK;
    const int blk = i / m.B;
    const int rt = pair_row(i, 0), rc = pair_row(i, 1);
    m.D[(size_t)i * 2 * RANK + d] = f2bf(m.dX[(size_t)rt * r3 + d] + m.dX[(size_t)rc * r3 + d]);
    float dug = 0.f;
    for (int jj = 0; jj < m.B; ++jj) {
        const int p = blk * m.B + jj;
        dug += m.dX[(size_t)pair_row(p, 0) * r3 + RANK + d] + m.dX[(size_t)pair_row(p, 1) * r3 + RANK + d];
    }
    m.D[(size_t)i * 2 * RANK + RANK + d] = f2bf(dug / (float)m.B);
    atomicAdd(m.gW_e + (size_t)m.xrow[rt] * RANK + d, m.dX[(size_t)rt * r3 + 2 * RANK + d]);
    atomicAdd(m.gW_e + (size_t)m.xrow[rc] * RANK + d, m.dX[(size_t)rc * r3 + 2 * RANK + d]);
}

}  // namespace xp
