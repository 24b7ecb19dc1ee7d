// accept_kernels.cu -- speculative acceptance of refined blocks (Sec. 3.1).
//
//   k_acc_rows    per target row (block position k = 1..B+1) and vocabulary
//                 chunk: argmax (T <= 0) or the running max / sum of exp of
//                 target / T (T > 0)
//   k_acc_decide  per block: the decision (greedy -- longest prefix equal to
//                 the target argmax plus the target's next token; lossless --
//                 accept y_k while u_k q_k(y_k) < p_k(y_k), q from the
//                 refinement pass (exp(l_y/T - lse)), p = softmax(target_k / T))
//                 and, for a sampling block, its draw descriptor
//                 (batches of at most ACCEPT_FUSED_MAX_B blocks skip this
//                 kernel: every CTA of k_acc_draw takes the decisions itself,
//                 which saves a dependent launch on the latency-bound path)
//   k_acc_draw    every draw of the batch over every vocabulary range:
//                 Gumbel-max over log max(0, p_k - q_k) at the first rejected
//                 position (q_k recomputed from z_final through W_r, read once
//                 per 32 draws), with the draw from p_k alongside for an empty
//                 residual, or the bonus draw from p_{B+1} after B acceptances;
//                 the last CTA emits the drawn tokens
#include "common.cuh"
#include "kernels.h"
#include "mlp_common.cuh"

namespace xp {

__device__ __forceinline__ Partial ldcg_partial16(const Partial *q)
{
    const float4 v = __ldcg(reinterpret_cast<const float4 *>(q));
    return Partial{v.x, __float_as_int(v.y), v.z, v.w};
}

// The running state of one thread over 16-byte pieces of a target row: T <= 0
// the first maximum; T > 0 the maximum in log2 units (y = x log2(e) / T) and
// the sum of 2^(y - max), rescaled once per batch of pieces.
template <int DT>
struct RowState {
    static constexpr int EP = DT ? 8 : 4;         // values per 16-byte piece
    float m, s;                                   // T <= 0: m the best value
    int idx;
    __device__ __forceinline__ void init() { m = -INFINITY; s = 0.0f; idx = 0x7fffffff; }
    static __device__ __forceinline__ void unpack(const uint4 &x, float (&v)[EP])
    {
        const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if constexpr (DT != 0) {
                v[2 * q] = __uint_as_float(w[q] << 16);
                v[2 * q + 1] = __uint_as_float(w[q] & 0xFFFF0000u);
            } else {
                v[q] = __uint_as_float(w[q]);
            }
        }
    }
    // one batch: U pieces of ids v, v + step, ... (n of them exist)
    template <int U>
    __device__ __forceinline__ void add(const uint4 (&x)[U], int n, int v, int step, float c2)
    {
        if constexpr (DT != 0) {
            // two bf16 per word: maxima on the words (exact; NaN loses), the rest in packed fp32
            constexpr uint32_t NEG2 = 0xFF80FF80u;         // two -inf
            if (c2 <= 0.0f) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (u >= n) break;
                    const uint32_t w = max_bf16x2(max_bf16x2(x[u].x, x[u].y), max_bf16x2(x[u].z, x[u].w));
                    const float m8 = fmaxf(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
                    if (m8 > m) {                     // the first id of the piece that holds it
                        float f[EP];
                        unpack(x[u], f);
                        int jj = EP - 1;
#pragma unroll
                        for (int j = EP - 2; j >= 0; --j)
                            if (f[j] == m8) jj = j;
                        m = m8;
                        idx = v + u * step + jj;
                    }
                }
                return;
            }
            uint32_t w2 = NEG2;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t w = max_bf16x2(max_bf16x2(x[u].x, x[u].y), max_bf16x2(x[u].z, x[u].w));
                w2 = max_bf16x2(w2, u < n ? w : NEG2);
            }
            const float mx = fmaxf(__uint_as_float(w2 << 16), __uint_as_float(w2 & 0xFFFF0000u));
            const float mn = fmaxf(m, mx * c2);       // c2 > 0 keeps the order
            const float ref = mn == -INFINITY ? 0.0f : mn;   // only masked values so far: every term is 2^-inf = 0
            const unsigned long long cc = f32x2(c2, c2), nr = f32x2(-ref, -ref);
            unsigned long long t[2] = {0, 0};
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (u >= n) break;
                const uint32_t w[4] = {x[u].x, x[u].y, x[u].z, x[u].w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float e0, e1;
                    f32x2_split(fma_f32x2(bf16x2_to_f32x2(w[q]), cc, nr), e0, e1);
                    t[q & 1] = add_f32x2(t[q & 1], f32x2(ex2_approx(e0), ex2_approx(e1)));
                }
            }
            float t0, t1;
            f32x2_split(add_f32x2(t[0], t[1]), t0, t1);
            s = s * ex2_approx(m - ref) + (t0 + t1);
            m = mn;
            return;
        }
        if (c2 <= 0.0f) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (u >= n) break;
                float f[EP];
                unpack(x[u], f);
                float m8 = f[0];
#pragma unroll
                for (int j = 1; j < EP; ++j) m8 = fmaxf(m8, f[j]);
                if (m8 > m) {                     // the first id of the piece that holds it
                    int jj = EP - 1;
#pragma unroll
                    for (int j = EP - 2; j >= 0; --j)
                        if (f[j] == m8) jj = j;
                    m = m8;
                    idx = v + u * step + jj;
                }
            }
            return;
        }
        float mb[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            float f[EP];
            unpack(x[u], f);
            float m8 = f[0];
#pragma unroll
            for (int j = 1; j < EP; ++j) m8 = fmaxf(m8, f[j]);
            mb[u] = u < n ? m8 : -INFINITY;
        }
        float mx = mb[0];
#pragma unroll
        for (int u = 1; u < U; ++u) mx = fmaxf(mx, mb[u]);
        const float mn = fmaxf(m, mx * c2);       // c2 > 0 keeps the order
        const float ref = mn == -INFINITY ? 0.0f : mn;   // only masked values so far: every term is 2^-inf = 0
        float t[2] = {0.0f, 0.0f};
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (u >= n) break;
            float f[EP];
            unpack(x[u], f);
#pragma unroll
            for (int j = 0; j < EP; ++j) t[j & 1] += ex2_approx(fmaf(f[j], c2, -ref));
        }
        s = s * ex2_approx(m - ref) + (t[0] + t[1]);
        m = mn;
    }
};

// Persistent grid of 256-thread CTAs (4 per SM); work item i = (target row
// i / chunks, vocabulary chunk i % chunks), dealt round-robin so that the CTAs
// stay evenly loaded (a large batch has many more items than resident CTAs);
// chunk boundaries are multiples of 8 ids, so every piece is whole (V % 8 == 0).
// The three kernels are chained with programmatic dependent launch: each of
// the first two lets the next one start early and every kernel waits
// (griddepcontrol.wait) for its predecessor's results right before reading
// them.  k_acc_rows reads only the target logits and temperatures, so it may
// run while the preceding kernel of the stream (the refinement) finishes; it
// waits for that kernel before it exits, so that the later kernels' waits
// cover it too.  It clears the status word and the draw counters.
//
// The pieces of a thread's next batch (four of 16 bytes, of the next item once the
// current one is used up) are requested before the current batch is reduced, so
// the loads do not wait for the arithmetic or for an item's merge, which costs five
// shuffle rounds and one barrier (double-buffered by item parity).  bf16 maxima are
// taken on the packed words and the exponentials' arguments and sums in packed
// fp32.  Measured under ncu at 2112 rows of 151936 bf16, half of them sampling: 219
// us with the loads of a batch issued after the previous batch's arithmetic and a
// shared-memory tree per item, 153 with batches ahead, 144 with the packed
// arithmetic; 544 sampling rows 66, 46, 43.  That is 4.5 and 3.8 TB/s, 0.67 and 0.58
// of the copy bandwidth, so HBM alone does not bound it: what is left is the mix of
// the exponentials' issue slots and of the bytes that registers hold in flight.
// Eight pieces and 3 CTAs an SM took 138 and 43 and made a call of one block 1 %
// slower; other cache hints change nothing.
namespace {

constexpr int ROWS_U = 4;                         // pieces in flight per thread and batch

template <int DT>
__device__ __forceinline__ void acc_rows_body(const AcceptParams &p, int chunks)
{
    constexpr int EP = RowState<DT>::EP, STEP = EP * 256;
    __shared__ Partial sp[2][8];
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int items = p.b * (p.B + 1) * chunks;
    const int V8 = p.V / 8;
    const char *target = static_cast<const char *>(p.target);
    // the cursor of the loads, one batch ahead of the arithmetic
    struct Cur { int item, v, v1; };
    auto open = [&](Cur &c) {
        if (c.item < items) {
            const int ch = c.item % chunks;
            c.v = 8 * (int)((long long)V8 * ch / chunks) + EP * threadIdx.x;
            c.v1 = 8 * (int)((long long)V8 * (ch + 1) / chunks);
        }
    };
    auto load = [&](const Cur &c, uint4 (&x)[ROWS_U]) {
        if (c.item >= items) return;
        const char *row = target + (size_t)(c.item / chunks) * p.V * (DT ? 2 : 4);
#pragma unroll
        for (int u = 0; u < ROWS_U; ++u)
            if (c.v + u * STEP < c.v1)
                x[u] = __ldg(reinterpret_cast<const uint4 *>(row + (size_t)(c.v + u * STEP) * (DT ? 2 : 4)));
    };
    Cur nx{(int)blockIdx.x, 0, 0};
    open(nx);
    uint4 xn[ROWS_U];
#pragma unroll
    for (int u = 0; u < ROWS_U; ++u) xn[u] = make_uint4(0, 0, 0, 0);
    load(nx, xn);
    int par = 0;
    float c2 = 0.0f;
    RowState<DT> st;
    st.init();
    bool fresh = true;
    while (nx.item < items) {
        const Cur cu = nx;
        uint4 x[ROWS_U];
#pragma unroll
        for (int u = 0; u < ROWS_U; ++u) x[u] = xn[u];
        // the next batch: of this item (every thread takes the same number of
        // batches, so that the CTA meets each item's barrier together), or the
        // first of the next one
        const int base = nx.v - EP * (int)threadIdx.x;
        const bool last = base + ROWS_U * STEP >= nx.v1;
        if (last) {
            nx.item += gridDim.x;
            open(nx);
        } else {
            nx.v += ROWS_U * STEP;
        }
        load(nx, xn);
        const int row = cu.item / chunks;         // seq * (B + 1) + k
        if (fresh) {
            const float T = p.temperature[row / (p.B + 1)];
            c2 = T > 0.0f ? (1.0f / T) * 1.4426950408889634f : 0.0f;
            fresh = false;
        }
        const int left = cu.v1 - cu.v;            // ids from this thread's first piece to the chunk's end
        const int n = left <= 0 ? 0 : min(ROWS_U, (left + STEP - 1) / STEP);
        if (n > 0) st.add(x, n, cu.v, STEP, c2);
        if (!last) continue;
        // the item's merge: warp, then CTA.  T > 0 in natural units from here on
        Partial a{-INFINITY, 0x7fffffff, -INFINITY, 0.0f};
        const bool sampling = c2 > 0.0f;
        if (!sampling) {
            a.best = st.m;
            a.idx = st.idx;
        } else if (st.m > -INFINITY) {
            a.m = st.m * 0.6931471805599453f;     // sum e^(x / T - m)
            a.s = st.s;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            Partial b;
            b.best = __shfl_xor_sync(0xffffffffu, a.best, o);
            b.idx = __shfl_xor_sync(0xffffffffu, a.idx, o);
            b.m = __shfl_xor_sync(0xffffffffu, a.m, o);
            b.s = __shfl_xor_sync(0xffffffffu, a.s, o);
            merge_partial(a, b, sampling);
        }
        if (lane == 0) sp[par][warp] = a;
        __syncthreads();
        if (threadIdx.x == 0) {
            a = sp[par][0];
            for (int w = 1; w < 8; ++w) merge_partial(a, sp[par][w], sampling);
            p.rowpart[(size_t)row * chunks + cu.item % chunks] = a;
        }
        par ^= 1;
        st.init();
        fresh = true;
    }
}

}  // namespace

__global__ void __launch_bounds__(256, 4) k_acc_rows(AcceptParams p, int chunks)
{
    pdl_trigger();
    if (blockIdx.x == 0) {
        if (threadIdx.x == 0) {
            *p.status = 0;
            p.ticket[0] = 0;                      // draws listed by k_acc_decide
            p.ticket[1] = 0;                      // CTAs of k_acc_draw done
        }
        for (int i = threadIdx.x; i < 2 * p.b; i += blockDim.x) p.keys[i] = 0ull;   // draw keys
    }
    if (p.dtype) acc_rows_body<1>(p, chunks);
    else acc_rows_body<0>(p, chunks);
    pdl_wait();
}

// One warp: the decision of block `seq`.  Lane k combines the chunk partials
// of target row k and decides position k (greedy: y_k equals the target
// argmax; lossless: u_k q_k(y_k) < p_k(y_k), q from the refinement pass,
// p = softmax(target_k / T)); a ballot finds the first position not
// accepted.  With `write`, the warp writes the accepted prefix, -1 past it
// and the accept length; a greedy block also the target's token after the
// prefix (a sampling block's token there is the draw's).  Returns whether the
// block samples and, for a sampling block, fills its draw descriptor (its
// rejected position, or B for the bonus draw).
__device__ __forceinline__ bool decide_block(const AcceptParams &p, int seq, int lane, Partial *rows, bool write,
                                             DrawDesc &dd)
{
    const int B = p.B, chunks = p.chunks;
    const float T = p.temperature[seq];
    const bool sampling = T > 0.0f;
    const float invT = sampling ? 1.0f / T : 0.0f;
    for (int k = lane; k <= B; k += 32) {
        Partial a{-INFINITY, 0x7fffffff, -INFINITY, 0.0f};
        const size_t r = (size_t)seq * (B + 1) + k;
        // eight chunks' partials requested together per round
        for (int c0 = 0; c0 < chunks; c0 += 8) {
            Partial q[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                q[u] = c0 + u < chunks ? ldcg_partial16(p.rowpart + r * chunks + c0 + u)
                                       : Partial{-INFINITY, 0x7fffffff, -INFINITY, 0.0f};
#pragma unroll
            for (int u = 0; u < 8; ++u) merge_partial(a, q[u], sampling);
        }
        rows[k] = a;
    }
    __syncwarp();
    int y = -1;
    bool ok = false;
    if (lane < B) {
        y = p.tokens[(size_t)seq * B + lane];
        if (y < 0 || y >= p.V) {
            set_status(p.status, ST_BOUNDS);
            y = 0;
        }
        if (!sampling) {
            ok = y == rows[lane].idx;
        } else {
            const int row = seq * (B + 1) + lane;
            const float lse_p = rows[lane].m + logf(rows[lane].s);
            const float p_y = expf(ld_any(p.target, p.dtype, (size_t)row * p.V + y) * invT - lse_p);
            const float q_y = expf(p.logit_sel[(size_t)seq * B + lane] - p.lse[(size_t)seq * B + lane]);
            const float u = uniform01(p.seed[seq], 0u, (uint32_t)lane, STREAM_ACCEPT, p.offset);
            ok = u * q_y < p_y;
        }
    }
    const unsigned rejected = __ballot_sync(0xffffffffu, lane < B && !ok);
    const int n = rejected ? __ffs(rejected) - 1 : B;
    if (write) {
        int32_t *out = p.out_tokens + (size_t)seq * (B + 1);
        for (int k = lane; k <= B; k += 32)
            if (k != n) out[k] = k < n ? p.tokens[(size_t)seq * B + k] : -1;
        if (lane == 0) {
            p.accept_len[seq] = n;
            if (!sampling) out[n] = rows[n].idx;
        }
    }
    if (sampling) {
        dd.seq = seq;
        dd.k = n;
        dd.invT = invT;
        dd.lse_p = rows[n].m + logf(rows[n].s);
        dd.lse_q = n < B ? p.lse[(size_t)seq * B + n] : 0.0f;
    }
    __syncwarp();                                 // rows is reused by the warp's next block
    return sampling;
}

// grid b, 32 threads (one warp per block): the block's decision
// (decide_block); a sampling block appends its draw descriptor for
// k_acc_draw.
__global__ void __launch_bounds__(32) k_acc_decide(AcceptParams p)
{
    pdl_trigger();                                // k_acc_draw may start its prologue
    pdl_wait();                                   // the row partials (and the refinement before them)
    __shared__ Partial rows[MAX_B + 1];
    DrawDesc dd{};
    if (decide_block(p, blockIdx.x, threadIdx.x, rows, true, dd) && threadIdx.x == 0) p.draws[atomicAdd(p.ticket, 1)] = dd;
}

// Small batches (fused): every CTA of the draw kernel takes all the
// decisions itself (warp w: blocks w, w + 8, ...), CTA 0 writes the accepted
// prefixes, and the sampling blocks' draw descriptors are listed in block
// order in shared memory (the same list in every CTA).  Returns their count.
__device__ __forceinline__ int decide_all(const AcceptParams &p, DrawDesc *list, Partial (*rows)[MAX_B + 1],
                                          int *sflag)
{
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, nwarps = blockDim.x / 32;
    for (int seq = warp; seq < p.b; seq += nwarps) {
        DrawDesc dd{};
        const bool s = decide_block(p, seq, lane, rows[warp], blockIdx.x == 0, dd);
        if (lane == 0) {
            sflag[seq] = s;
            if (s) list[seq] = dd;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int nd = 0;
        for (int seq = 0; seq < p.b; ++seq)
            if (sflag[seq]) list[nd++] = list[seq];
        sflag[ACCEPT_FUSED_MAX_B] = nd;
    }
    __syncthreads();
    return sflag[ACCEPT_FUSED_MAX_B];
}

namespace {
constexpr int DRAW_NZ = 16;         // fp32: draws per sweep of the vocabulary (accumulators per lane)
constexpr int DRAW_THREADS = 256;

// 32 consecutive elements of row v of the fp32 W_r.
__device__ __forceinline__ void load_row32(float (&w)[32], const void *W_r, bool al, int v, int k0)
{
    const float *src = static_cast<const float *>(W_r) + (size_t)v * RANK + k0;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const float4 x = ld4(src + 4 * c, al);
        w[4 * c] = x.x; w[4 * c + 1] = x.y; w[4 * c + 2] = x.z; w[4 * c + 3] = x.w;
    }
}
}  // namespace

// The end of the draw kernel, every thread of every CTA: the CTA counts
// itself done; the last one emits each drawn token (the residual's draw, or
// the draw from p when the residual is empty or after B acceptances).
__device__ __forceinline__ void draw_finish(const AcceptParams &p, const DrawDesc *list, int nd, int G, int *s_last)
{
    if (threadIdx.x == 0) {
        __threadfence();
        *s_last = atomicAdd(p.ticket + 1, 1) == G - 1;
    }
    __syncthreads();
    if (!*s_last) return;
    __threadfence();
    for (int j = threadIdx.x; j < nd; j += blockDim.x) {
        const DrawDesc dd = list[j];
        const unsigned long long kr = __ldcg(p.keys + 2 * dd.seq), kp = __ldcg(p.keys + 2 * dd.seq + 1);
        float best;
        int idx;
        argmax_unkey(dd.k < p.B && kr ? kr : kp, best, idx);
        p.out_tokens[(size_t)dd.seq * (p.B + 1) + dd.k] = idx;
    }
}

// Scores of one (draw, vocabulary id) pair, merged into the lane's running
// bests: the p draw tx + g, and for a residual draw log(max(0, p - q)) + g
// with l = acc + s recomputed (acc = (W_r z)_v).
__device__ __forceinline__ void draw_element(const AcceptParams &p, const DrawDesc &dd, unsigned long long seed, int v,
                                             float acc, float g, float &rb, int &ri, float &pb, int &pi)
{
    const size_t trow = (size_t)dd.seq * (p.B + 1) + dd.k;
    const float tx = ld_any(p.target, p.dtype, trow * p.V + v) * dd.invT;
    merge_argmax(pb, pi, tx + g, v);
    if (dd.k < p.B) {
        const float lx = (acc + ld_any(p.s, p.dtype, ((size_t)dd.seq * p.B + dd.k) * p.V + v)) * dd.invT;
        const float res = expf(tx - dd.lse_p) - expf(lx - dd.lse_q);
        if (res > 0.0f) merge_argmax(rb, ri, logf(res) + g, v);
    }
}

// grid G, 256 threads; CTA r owns the vocabulary range [V r / G, V (r+1) / G).
// Every draw of the batch (one per sampling block, listed by k_acc_decide) is
// taken over every range: Gumbel-max over log max(0, p_k - q_k) at the first
// rejected position k (q_k recomputed from z_final through W_r: each lane owns
// one vocabulary row and takes its dot products with the z of up to 16 draws
// held in shared memory, so W_r is read once per 16 draws), with the draw from
// p_k alongside for an empty residual, or the bonus draw from p_{B+1} after B
// acceptances.  Each range's best keys meet through 64-bit atomicMax (the
// fp32 score made order-preserving, then the inverted id: ties go to the
// smallest id); the last CTA to finish emits every drawn token.
//
// This is the last kernel of an acceptance call and it never triggers its
// dependents early (no griddepcontrol.launch_dependents): the next call's
// k_acc_rows, which may reuse the same scratch (always, for
// xpress_accept_noalloc), clears the counters before its own dependency wait,
// so it must not start until every CTA of this kernel has exited.
__global__ void __launch_bounds__(DRAW_THREADS) k_acc_draw_simt(AcceptParams p)
{
    pdl_wait();                                   // the draw list of k_acc_decide (or the row partials)
    __shared__ DrawDesc flist[ACCEPT_FUSED_MAX_B];
    __shared__ Partial frows[DRAW_THREADS / 32][MAX_B + 1];
    __shared__ int fflag[ACCEPT_FUSED_MAX_B + 1];
    const int nd = p.fused ? decide_all(p, flist, frows, fflag) : __ldcg(p.ticket);
    const DrawDesc *list = p.fused ? flist : p.draws;
    if (nd == 0) return;
    const int G = gridDim.x, r = blockIdx.x, warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int nwarps = DRAW_THREADS / 32, B = p.B;
    const int v0 = (int)((long long)p.V * r / G), v1 = (int)((long long)p.V * (r + 1) / G);
    __shared__ __align__(16) float zs[DRAW_NZ][RANK];   // read as float4
    __shared__ DrawDesc dsc[DRAW_NZ];
    __shared__ unsigned long long wkey[DRAW_THREADS / 32][DRAW_NZ][2];
    __shared__ int s_any_resid, s_last;
    const bool wal = al16(p.W_r);
    for (int g0 = 0; g0 < nd; g0 += DRAW_NZ) {
        const int nz = min(DRAW_NZ, nd - g0);
        if (threadIdx.x < nz) dsc[threadIdx.x] = list[g0 + threadIdx.x];
        if (threadIdx.x == 0) s_any_resid = 0;
        __syncthreads();
        for (int i = threadIdx.x; i < nz * RANK; i += DRAW_THREADS) {
            const int j = i / RANK, d = i % RANK;
            const DrawDesc dd = dsc[j];
            const bool resid = dd.k < B;
            zs[j][d] = resid ? round_op(p.z_final[((size_t)dd.seq * B + dd.k) * RANK + d], p.dtype) : 0.0f;
            if (resid && d == 0) s_any_resid = 1;
        }
        __syncthreads();
        const bool any_resid = s_any_resid != 0;
        float rb[DRAW_NZ], pb[DRAW_NZ];
        int ri[DRAW_NZ], pi[DRAW_NZ];
#pragma unroll
        for (int j = 0; j < DRAW_NZ; ++j) { rb[j] = pb[j] = -INFINITY; ri[j] = pi[j] = 0x7fffffff; }
        for (int vb = v0 + warp * 32; vb < v1; vb += nwarps * 32) {
            const int v = vb + lane;
            const bool valid = v < v1;
            float acc[DRAW_NZ];
#pragma unroll
            for (int j = 0; j < DRAW_NZ; ++j) acc[j] = 0.0f;
            if (any_resid && valid) {
#pragma unroll 1
                for (int k0 = 0; k0 < RANK; k0 += 32) {
                    float w[32];
                    load_row32(w, p.W_r, wal, v, k0);
#pragma unroll
                    for (int j = 0; j < DRAW_NZ; ++j) {
                        if (j < nz) {
                            const float4 *zz = reinterpret_cast<const float4 *>(&zs[j][k0]);
                            float a = acc[j];
#pragma unroll
                            for (int c = 0; c < 8; ++c) {
                                const float4 z4 = zz[c];
                                a = fmaf(w[4 * c], z4.x, a);
                                a = fmaf(w[4 * c + 1], z4.y, a);
                                a = fmaf(w[4 * c + 2], z4.z, a);
                                a = fmaf(w[4 * c + 3], z4.w, a);
                            }
                            acc[j] = a;
                        }
                    }
                }
            }
            if (valid) {
#pragma unroll
                for (int j = 0; j < DRAW_NZ; ++j) {
                    if (j < nz) {
                        const DrawDesc dd = dsc[j];
                        const unsigned long long seed = p.seed[dd.seq];
                        const float g = gumbel(seed, (uint32_t)v, (uint32_t)dd.k, STREAM_RESID, p.offset);
                        draw_element(p, dd, seed, v, acc[j], g, rb[j], ri[j], pb[j], pi[j]);
                    }
                }
            }
        }
        // warp, then CTA, then grid (atomicMax of the 64-bit keys)
#pragma unroll
        for (int j = 0; j < DRAW_NZ; ++j) {
            if (j < nz) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    merge_argmax(rb[j], ri[j], __shfl_xor_sync(0xffffffffu, rb[j], o),
                                 __shfl_xor_sync(0xffffffffu, ri[j], o));
                    merge_argmax(pb[j], pi[j], __shfl_xor_sync(0xffffffffu, pb[j], o),
                                 __shfl_xor_sync(0xffffffffu, pi[j], o));
                }
                if (lane == 0) {
                    wkey[warp][j][0] = ri[j] != 0x7fffffff ? argmax_key(rb[j], ri[j]) : 0ull;
                    wkey[warp][j][1] = pi[j] != 0x7fffffff ? argmax_key(pb[j], pi[j]) : 0ull;
                }
            }
        }
        __syncthreads();
        if (threadIdx.x < 2 * nz) {
            const int j = threadIdx.x >> 1, h = threadIdx.x & 1;
            unsigned long long k = 0ull;
            for (int w = 0; w < nwarps; ++w) k = wkey[w][j][h] > k ? wkey[w][j][h] : k;
            if (k) atomicMax(p.keys + 2 * dsc[j].seq + h, k);
        }
        __syncthreads();
    }
    draw_finish(p, list, nd, G, &s_last);
}


// bf16 refiners: the same draws with the residual's products W_r z on tensor
// cores (warp-level m16n8k16): 16 draws are the M rows, 8 vocabulary rows the N
// columns, K = r.  Any permutation of K applied to both operands leaves the
// products unchanged; lane (g, t) takes, for each 32-wide K slab, the 16-byte
// piece [8t, 8t + 8) of vocabulary row g as the B fragments of two k-steps, and
// the A fragments follow the same order.  Lane (g, t) then owns draws g and
// g + 8 at rows 2t and 2t + 1 of the 8, whose Gumbel noise comes from one
// Philox call.  CTA ranges start and end at multiples of 8 ids (V % 8 == 0).
//
// One CTA per SM: a copy warp streams the CTA's rows of W_r in 120-row blocks
// (60 KB, one bulk copy each: the rows are contiguous) through a 3-stage ring,
// 15 warps take 8 rows of a block each, for up to 32 draws a sweep.  Per (draw,
// id) the arithmetic (half a Philox call, four logarithms, two exponentials) is
// about 150 instructions, and 32 draws read W_r and 64 rows of s and target, so
// at the Qwen3-8B vocabulary both bounds lie near 20 us; what the kernel loses
// is latency and issue slots.  Hence the ring starts before the row statistics
// are complete (W_r does not depend on them), the s and target words of a
// warp's next block are requested before the current block's arithmetic, and
// the precise logarithms and exponentials are taken only for pairs that can
// still reach the best score of the CTA's warps (draw_candidate: a bound from
// two fast logarithms, the same winner).  Measured under
// ncu at 32 draws of 151936 ids: 52 us, against 102 us with each warp
// loading its 8 rows of W_r, then its s and target words, in turn (two CTAs of
// 8 warps per SM, 16 draws a sweep); 30 us against 37 us at 3 draws.
namespace {

constexpr int DW_WARPS = 15;                             // with the copy warp 512 threads: 128 registers each
constexpr int DW_THREADS = 32 * (DW_WARPS + 1);          // + the copy warp
constexpr int DW_ROWS = 8 * DW_WARPS;                    // vocabulary rows per block
constexpr uint32_t DW_BLOCK = DW_ROWS * RANK * 2;        // 60 KB
constexpr int DW_STAGES = 3;
constexpr int DW_NZ = 32;                                // draws per sweep
constexpr int DW_ZP = RANK + 32;                         // bf16 row pitch of the z operands: 16-byte reads of 8 lanes
                                                         // (2 rows x 4 pieces) meet 8 different bank groups

struct DrawShared {
    uint16_t zb[DW_NZ][DW_ZP];                           // first: 16-byte aligned
    union {
        unsigned long long wkey[DW_WARPS][DW_NZ][2];     // the sweep's best keys per warp
        Partial rows[DW_WARPS + 1][MAX_B + 1];           // decide_all (before the first sweep)
    };
    unsigned long long dseed[DW_NZ];
    uint32_t best[DW_NZ][2];                             // best p / residual score of any warp (order_key)
    uint64_t full[DW_STAGES], empty[DW_STAGES];
    DrawDesc dsc[DW_NZ];
    DrawDesc flist[ACCEPT_FUSED_MAX_B];
    int fflag[ACCEPT_FUSED_MAX_B + 1];
    int last, abort;
};

constexpr size_t DW_SMEM = 128 + DW_STAGES * DW_BLOCK + sizeof(DrawShared);
static_assert(DW_SMEM <= 232448, "k_acc_draw shared memory");

// The bf16 values of ids v and v + 1 (v even) of a row, as one word.
__device__ __forceinline__ uint32_t ld_pair(const void *base, size_t i, bool aligned4)
{
    const uint16_t *q = static_cast<const uint16_t *>(base) + i;
    if (aligned4) return __ldg(reinterpret_cast<const uint32_t *>(q));
    return (uint32_t)__ldg(q) | ((uint32_t)__ldg(q + 1) << 16);
}

// The value part of an argmax key: an order-preserving word of a float.
__device__ __forceinline__ uint32_t order_key(float x)
{
    const uint32_t b = __float_as_uint(x);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float order_unkey(uint32_t u)
{
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7FFFFFFFu) : ~u);
}

// Whether the pair of target value tv and uniform u can still win one of the
// two draws whose best scores so far (of any warp of the CTA) are pbest and
// rbest; false only if neither score can reach them.  With e = -log u >= 2^-9
// the fast logarithm (absolute error below 2^-21 on [1/2, 2], a few ulp
// elsewhere) gives the Gumbel noise to 2^-21 / 2^-9 and a few ulp, below the
// margin of 1e-3 (and 1e-5 of the score for the roundings of a large one);
// smaller e always count as candidates.  The draw from p of a rejected
// position is only taken when its residual is empty, so it no longer counts
// once the residual has a score (need_p).  The residual's score is at most the
// one of p alone, log(max(0, p - q)) <= log p = tx - lse_p, up to the rounding
// of an exponential, a factor of e at most where p is subnormal.
__device__ __forceinline__ bool draw_candidate(float invT, float lse_p, bool resid, bool need_p, float tv, float u,
                                               float pbest, float rbest)
{
    const float e = -__logf(u);
    const float tx = tv * invT, ps = tx - __logf(e);
    const float margin = fminf(fmaf(fabsf(ps) + fabsf(lse_p), 1e-5f, 1e-3f), 1e30f);
    const float rs = ps - lse_p + (tx - lse_p < -87.0f ? 1.0f : 0.0f);
    return e < 0.001953125f || (need_p && !(ps + margin < pbest)) || (resid && !(rs + margin < rbest));
}

__device__ __forceinline__ float word_uniform(uint32_t w) { return ((float)(w >> 9) + 0.5f) * (1.0f / 8388608.0f); }

// Scores of one (draw, vocabulary id) pair from its target and s values
// (draw_element with the values in hand).
__device__ __forceinline__ void draw_score(const DrawDesc &dd, bool resid, int v, float tv, float sv, float acc, float u,
                                           float &rb, int &ri, float &pb, int &pi)
{
    const float g = -logf(-logf(u));
    const float tx = tv * dd.invT;
    merge_argmax(pb, pi, tx + g, v);
    if (resid) {
        const float lx = (acc + sv) * dd.invT;
        const float res = expf(tx - dd.lse_p) - expf(lx - dd.lse_q);
        if (res > 0.0f) merge_argmax(rb, ri, logf(res) + g, v);
    }
}

}  // namespace

const size_t kAccDrawSmemBytes = DW_SMEM;
const int kAccDrawThreads = DW_THREADS;

__global__ void __launch_bounds__(DW_THREADS, 1) k_acc_draw(AcceptParams p)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *ring = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
    DrawShared &sh = *reinterpret_cast<DrawShared *>(ring + DW_STAGES * DW_BLOCK);
    const int G = gridDim.x, r = blockIdx.x, warp = threadIdx.x / 32, lane = threadIdx.x % 32, B = p.B;
    const int V8 = p.V / 8;
    const int v0 = 8 * (int)((long long)V8 * r / G), v1 = 8 * (int)((long long)V8 * (r + 1) / G);
    const int nblk = (v1 - v0 + DW_ROWS - 1) / DW_ROWS;
    const uint16_t *wr = static_cast<const uint16_t *>(p.W_r);
    volatile int *abort = &sh.abort;
    const bool copier = warp == DW_WARPS;
    if (threadIdx.x == 0) {
        for (int i = 0; i < DW_STAGES; ++i) {
            mbar_init(&sh.full[i], 1);
            mbar_init(&sh.empty[i], DW_WARPS);
        }
        sh.abort = 0;
        fence_barrier_init();
    }
    __syncthreads();
    auto issue = [&](int n) {                     // copies block n % nblk into stage n % DW_STAGES
        const int vb = v0 + (n % nblk) * DW_ROWS, st = n % DW_STAGES;
        const uint32_t bytes = (uint32_t)min(DW_ROWS, v1 - vb) * RANK * 2;
        mbar_expect_tx(&sh.full[st], bytes);
        bulk_load_1d(ring + st * DW_BLOCK, wr + (size_t)vb * RANK, bytes, &sh.full[st]);
    };
    int issued = 0;
    if (copier) {
        // a sampling block means a draw: start on W_r before the row statistics are complete
        bool any = false;
        for (int q = lane; q < p.b; q += 32) any = any || p.temperature[q] > 0.0f;
        any = __any_sync(0xffffffffu, any);
        if (lane == 0 && any)
            while (issued < min(DW_STAGES, nblk)) issue(issued++);
    }
    pdl_wait();                                   // the draw list of k_acc_decide (or the row partials)
    const int nd = p.fused ? decide_all(p, sh.flist, sh.rows, sh.fflag) : __ldcg(p.ticket);
    const DrawDesc *list = p.fused ? sh.flist : p.draws;
    const int total = nblk * ((nd + DW_NZ - 1) / DW_NZ);
    if (copier) {
        if (lane == 0) {
            for (; issued < total; ++issued)
                if (!mbar_wait(&sh.empty[issued % DW_STAGES], (uint32_t)(((issued / DW_STAGES) & 1) ^ 1), abort)) break;
                else issue(issued);
            if (*abort || total < issued) {
                // no copy may still be landing when the CTA leaves
                int dummy = 0;
                for (int n = max(0, issued - DW_STAGES); n < issued; ++n)
                    mbar_wait(&sh.full[n % DW_STAGES], (uint32_t)((n / DW_STAGES) & 1), &dummy, 100000000ull);
            }
        }
    } else {
        const int g = lane >> 2, tq = lane & 3;
        const bool al_t = (reinterpret_cast<uintptr_t>(p.target) & 3) == 0, al_s = (reinterpret_cast<uintptr_t>(p.s) & 3) == 0;
        int n = 0;
        for (int g0 = 0; g0 < nd; g0 += DW_NZ) {
            const int nz = min(DW_NZ, nd - g0);
            warps_bar<32 * DW_WARPS>();           // the previous sweep's keys (or the decisions) are read
            // one warp per draw: its descriptor and its z operand
            for (int j = warp; j < DW_NZ; j += DW_WARPS) {
                DrawDesc dd{};
                dd.k = B;                         // padding draws: no residual, never scored
                if (j < nz) dd = list[g0 + j];
                float z[RANK / 32];
#pragma unroll
                for (int i = 0; i < RANK / 32; ++i)
                    z[i] = dd.k < B ? p.z_final[((size_t)dd.seq * B + dd.k) * RANK + 32 * i + lane] : 0.0f;
#pragma unroll
                for (int i = 0; i < RANK / 32; ++i) sh.zb[j][32 * i + lane] = f2bf(z[i]);
                if (lane == 0) {
                    sh.dsc[j] = dd;
                    sh.dseed[j] = j < nz ? p.seed[dd.seq] : 0ull;
                    sh.best[j][0] = sh.best[j][1] = order_key(-INFINITY);
                }
            }
            warps_bar<32 * DW_WARPS>();
            // the target and s words of this lane's draws (16 q + g + 8 h) at ids v, v + 1
            uint32_t tw[2][2], sw[2][2];
            auto fetch = [&](int vb) {
                const int v = vb + 2 * tq;
#pragma unroll
                for (int q = 0; q < 2; ++q)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int j = 16 * q + g + 8 * h;
                        tw[q][h] = sw[q][h] = 0;
                        if (j < nz && vb < v1) {
                            const DrawDesc &dd = sh.dsc[j];
                            tw[q][h] = ld_pair(p.target, ((size_t)dd.seq * (B + 1) + dd.k) * p.V + v, al_t);
                            if (dd.k < B) sw[q][h] = ld_pair(p.s, ((size_t)dd.seq * B + dd.k) * p.V + v, al_s);
                        }
                    }
            };
            float rb[2][2], pb[2][2];
            int ri[2][2], pi[2][2];
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    rb[q][h] = pb[q][h] = -INFINITY;
                    ri[q][h] = pi[q][h] = 0x7fffffff;
                }
            bool ok = true;
            fetch(v0 + 8 * warp);
            for (int bi = 0; bi < nblk; ++bi, ++n) {
                const int vb = v0 + bi * DW_ROWS + 8 * warp, st = n % DW_STAGES;
                uint32_t tc[2][2], sc[2][2];
#pragma unroll
                for (int q = 0; q < 2; ++q)
#pragma unroll
                    for (int h = 0; h < 2; ++h) { tc[q][h] = tw[q][h]; sc[q][h] = sw[q][h]; }
                fetch(vb + DW_ROWS);
                if (!mbar_wait_warp(&sh.full[st], (uint32_t)((n / DW_STAGES) & 1), abort)) { ok = false; break; }
                uint4 w[RANK / 32];
                const uint8_t *src = ring + st * DW_BLOCK + (8 * warp + g) * (RANK * 2) + 16 * tq;
                if (vb < v1) {
#pragma unroll
                    for (int s = 0; s < RANK / 32; ++s) w[s] = *reinterpret_cast<const uint4 *>(src + 64 * s);
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.empty[st]);
                if (vb >= v1) continue;
                const int v = vb + 2 * tq;
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    if (16 * q >= nz) break;
                    float c[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                    __syncwarp();             // the scores of the 16 draws before are taken lane by lane
#pragma unroll
                    for (int s = 0; s < RANK / 32; ++s) {
                        // physical columns 32 s + 8 t + {0, 1 | 2, 3} are k-step 2 s, + {4, 5 | 6, 7} k-step 2 s + 1
                        const uint4 a0 = *reinterpret_cast<const uint4 *>(&sh.zb[16 * q + g][32 * s + 8 * tq]);
                        const uint4 a1 = *reinterpret_cast<const uint4 *>(&sh.zb[16 * q + g + 8][32 * s + 8 * tq]);
                        const uint32_t f0[4] = {a0.x, a1.x, a0.y, a1.y}, f1[4] = {a0.z, a1.z, a0.w, a1.w};
                        mma_bf16_16816(c, f0, w[s].x, w[s].y);
                        mma_bf16_16816(c, f1, w[s].z, w[s].w);
                    }
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int j = 16 * q + g + 8 * h;
                        if (j < nz) {
                            const DrawDesc &dd = sh.dsc[j];
                            const bool resid = dd.k < B;
                            const unsigned long long seed = sh.dseed[j];
                            const uint4 o = philox10(make_uint4((uint32_t)v >> 2, (uint32_t)dd.k, STREAM_RESID, p.offset),
                                                     (uint32_t)seed, (uint32_t)(seed >> 32));
                            // v is even: one Philox call gives both ids' words
                            const float u0 = word_uniform((v & 2) ? o.z : o.x), u1 = word_uniform((v & 2) ? o.w : o.y);
                            const float t0 = __uint_as_float(tc[q][h] << 16), t1 = __uint_as_float(tc[q][h] & 0xFFFF0000u);
                            const volatile uint32_t *sb = sh.best[j];
                            const float pl = fmaxf(pb[q][h], order_unkey(sb[0])), rl = fmaxf(rb[q][h], order_unkey(sb[1]));
                            const bool need_p = !resid || rl == -INFINITY;
                            const bool c0 = draw_candidate(dd.invT, dd.lse_p, resid, need_p, t0, u0, pl, rl);
                            const bool c1 = draw_candidate(dd.invT, dd.lse_p, resid, need_p, t1, u1, pl, rl);
                            if (c0 || c1) {
                                if (c0)
                                    draw_score(dd, resid, v, t0, __uint_as_float(sc[q][h] << 16), c[2 * h], u0, rb[q][h],
                                               ri[q][h], pb[q][h], pi[q][h]);
                                if (c1)
                                    draw_score(dd, resid, v + 1, t1, __uint_as_float(sc[q][h] & 0xFFFF0000u), c[2 * h + 1],
                                               u1, rb[q][h], ri[q][h], pb[q][h], pi[q][h]);
                                if (pb[q][h] > pl) atomicMax(&sh.best[j][0], order_key(pb[q][h]));
                                if (rb[q][h] > rl) atomicMax(&sh.best[j][1], order_key(rb[q][h]));
                            }
                        }
                    }
                }
            }
            // the four lanes of a row group share their draws: reduce over t
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
#pragma unroll
                    for (int o = 1; o <= 2; o <<= 1) {
                        merge_argmax(rb[q][h], ri[q][h], __shfl_xor_sync(0xffffffffu, rb[q][h], o),
                                     __shfl_xor_sync(0xffffffffu, ri[q][h], o));
                        merge_argmax(pb[q][h], pi[q][h], __shfl_xor_sync(0xffffffffu, pb[q][h], o),
                                     __shfl_xor_sync(0xffffffffu, pi[q][h], o));
                    }
                    if (tq == 0) {
                        const int j = 16 * q + g + 8 * h;
                        sh.wkey[warp][j][0] = ri[q][h] != 0x7fffffff ? argmax_key(rb[q][h], ri[q][h]) : 0ull;
                        sh.wkey[warp][j][1] = pi[q][h] != 0x7fffffff ? argmax_key(pb[q][h], pi[q][h]) : 0ull;
                    }
                }
            if (warps_bar_or<32 * DW_WARPS>(!ok || *abort)) break;
            if ((int)threadIdx.x < 2 * nz) {
                const int j = threadIdx.x >> 1, hh = threadIdx.x & 1;
                unsigned long long k = 0ull;
                for (int w2 = 0; w2 < DW_WARPS; ++w2) k = sh.wkey[w2][j][hh] > k ? sh.wkey[w2][j][hh] : k;
                if (k) atomicMax(p.keys + 2 * sh.dsc[j].seq + hh, k);
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && sh.abort) set_status(p.status, ST_TIMEOUT);
    if (nd > 0) draw_finish(p, list, nd, G, &sh.last);
}

}  // namespace xp
