// Adaptive layer fusion (Eq. 3, Sec. 4.1) and the bookkeeping of a context append.
//
// fusion_alpha: alpha^(i) = softmax(W^fuse_{i,:}), computed once when the weights are set
// (Sec. 4.1: the normalised weights can be cached after training).
// fuse_layers: the T target rows of every new position are read once and every draft layer's
// fused, normalised row is written: a thread-block cluster per position for a handful of
// positions (one block step), one CTA per position when there are enough to fill the GPU
// (context fill).
#include <math.h>

#include <algorithm>
#include <type_traits>

#include <cooperative_groups.h>

#include "common.cuh"
#include "internal.h"
#include "umma.cuh"

namespace cg = cooperative_groups;

namespace dfl {
namespace {

__global__ void fusion_alpha_kernel(const float* __restrict__ w, float* __restrict__ alpha, int D,
                                    int T, int raw) {
    pdl_trigger();
    pdl_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= D) return;
    const float* row = w + (size_t)i * T;
    if (raw) {
        for (int j = 0; j < T; ++j) alpha[(size_t)i * T + j] = row[j];
        return;
    }
    float m = -INFINITY;
    for (int j = 0; j < T; ++j) m = fmaxf(m, row[j]);
    float s = 0.f;
    for (int j = 0; j < T; ++j) s += expf(row[j] - m);
    for (int j = 0; j < T; ++j) alpha[(size_t)i * T + j] = expf(row[j] - m) / s;
}

__global__ void fuse_begin_kernel(int32_t* ctx_len, int32_t* app_base, int32_t* app_cnt,
                                  const int32_t* __restrict__ n_new, int batch, int n_max,
                                  int max_ctx, uint32_t* err) {
    pdl_trigger();
    pdl_wait();
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= batch) return;
    const int L = ctx_len[b];
    int n = n_new[b];
    if (n < 0 || n > n_max || L + n > max_ctx) {
        atomicOr(err, DFLARE_DEVERR_CAPACITY);
        n = 0;
    }
    app_base[b] = L;
    app_cnt[b] = n;
    ctx_len[b] = L + n;
}

constexpr int kFuseCH = 512;       // features per CTA (64 threads x 8)
constexpr int kFuseGroups = 4;     // thread groups splitting the T target layers

// One position is handled by a cluster of ceil(d / 512) CTAs (at most 8 for d <= 4096); CTA c owns
// features [512 c, 512 c + 512). Each CTA (256 threads) stages its slice of all T target rows and
// of the D gain rows in shared memory with cp.async (one round trip). Thread group q (64 threads,
// 8 features each) forms the D weighted sums over target layers j = q, q + 4, ...; the four
// partial sums are added in group order, the CTA reduces its partial sums of squares, and the
// CTAs of the cluster exchange those partials through distributed shared memory (one gather,
// summed in rank order) before normalising.
template <class T, int DMAX>
__global__ void __launch_bounds__(256) fuse_layers_kernel(
    const T* __restrict__ H, const float* __restrict__ alpha, const T* __restrict__ gain,
    T* __restrict__ F, T* __restrict__ F_out, const int32_t* __restrict__ app_cnt, int D, int Tn,
    int batch, int n_max, int d, long long f_layer_rows, float eps) {
    pdl_trigger();
    pdl_wait();
    extern __shared__ __align__(16) uint8_t smem[];
    T* sh = reinterpret_cast<T*>(smem);          // [Tn][kFuseCH] target rows, then [D][kFuseCH] gains
    T* sg = sh + (size_t)Tn * kFuseCH;
    float* sacc = reinterpret_cast<float*>(sg + (size_t)D * kFuseCH);  // [3][DMAX][8][64]
    __shared__ float s_alpha[16 * 64];
    __shared__ float red[2][DMAX];
    __shared__ float ss_cta[DMAX];               // this CTA's partial sums of squares
    __shared__ float part[8][DMAX];              // every cluster rank's partials
    __shared__ float inv_s[DMAX];
    cg::cluster_group cluster = cg::this_cluster();
    const int C = (int)cluster.num_blocks(), cr = (int)cluster.block_rank();
    const int r = blockIdx.y, b = blockIdx.z;
    if (r >= app_cnt[b]) return;                 // the same for every CTA of the cluster
    const int tid = threadIdx.x, q = tid >> 6, t64 = tid & 63;
    const int lane = tid & 31, warp = tid >> 5;
    const int f0 = cr * kFuseCH, nf = min(kFuseCH, d - f0);
    const size_t row = (size_t)b * n_max + r;
    const size_t lstride = (size_t)batch * n_max * d;
    constexpr int EPC = 16 / sizeof(T);          // elements per 16-byte copy
    const int per_row = nf / EPC;                // <= 64 (bf16) or 128 (fp32)
    const uint32_t ssh = (uint32_t)__cvta_generic_to_shared(sh);
    // all T target rows of this slice and all D gain rows, one round trip
    for (int j = q; j < Tn + D; j += kFuseGroups) {
        const T* src = j < Tn ? H + (size_t)j * lstride + row * d + f0 : gain + (size_t)(j - Tn) * d + f0;
        for (int p = t64; p < per_row; p += 64)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                             ssh + (uint32_t)((j * kFuseCH + p * EPC) * sizeof(T))),
                         "l"(src + p * EPC)
                         : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    for (int k = tid; k < D * Tn; k += blockDim.x) s_alpha[k] = alpha[k];
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    const int e0 = t64 * 8;
    const bool act = e0 < nf;
    for (int i0 = 0; i0 < D; i0 += DMAX) {
        const int nd = min(DMAX, D - i0);
        float acc[DMAX][8];
#pragma unroll
        for (int i = 0; i < DMAX; ++i)
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[i][e] = 0.f;
        if (act) {
            for (int j = q; j < Tn; j += kFuseGroups) {
                float h[8], a[DMAX];
                load8(sh + j * kFuseCH + e0, h);
#pragma unroll
                for (int i = 0; i < DMAX; ++i) a[i] = i < nd ? s_alpha[(i0 + i) * Tn + j] : 0.f;
#pragma unroll
                for (int i = 0; i < DMAX; ++i)
#pragma unroll
                    for (int e = 0; e < 8; ++e) acc[i][e] = fmaf(a[i], h[e], acc[i][e]);
            }
        }
        // groups 1..3 hand their partial sums to group 0, which adds them in group order
        if (q > 0) {
#pragma unroll
            for (int i = 0; i < DMAX; ++i)
#pragma unroll
                for (int e = 0; e < 8; ++e) sacc[(((q - 1) * DMAX + i) * 8 + e) * 64 + t64] = acc[i][e];
        }
        __syncthreads();
        if (q == 0) {
#pragma unroll
            for (int g2 = 0; g2 < kFuseGroups - 1; ++g2)
#pragma unroll
                for (int i = 0; i < DMAX; ++i)
#pragma unroll
                    for (int e = 0; e < 8; ++e) acc[i][e] += sacc[((g2 * DMAX + i) * 8 + e) * 64 + t64];
#pragma unroll
            for (int i = 0; i < DMAX; ++i) {
                float v = 0.f;
#pragma unroll
                for (int e = 0; e < 8; ++e) v = fmaf(acc[i][e], acc[i][e], v);
                v = warp_sum(v);
                if (lane == 0) red[warp][i] = v;
            }
        }
        __syncthreads();
        if (tid < DMAX) ss_cta[tid] = red[0][tid] + red[1][tid];
        cluster.sync();
        // gather every rank's partials in one round of DSMEM loads, then sum in rank order
        for (int k = tid; k < C * nd; k += blockDim.x)
            part[k / nd][k % nd] = cluster.map_shared_rank(ss_cta, k / nd)[k % nd];
        __syncthreads();
        if (tid < nd) {
            float tot = 0.f;
            for (int c = 0; c < C; ++c) tot += part[c][tid];
            inv_s[tid] = inv_rms(tot, d, eps);
        }
        __syncthreads();
        if (q == 0 && act) {
#pragma unroll
            for (int i = 0; i < DMAX; ++i) {
                if (i >= nd) break;
                float g[8], o[8];
                load8(sg + (i0 + i) * kFuseCH + e0, g);
                const float inv = inv_s[i];
#pragma unroll
                for (int e = 0; e < 8; ++e) o[e] = g[e] * (acc[i][e] * inv);
                store8(F + ((size_t)(i0 + i) * f_layer_rows + row) * d + f0 + e0, o);
                if (F_out)
                    store8(F_out + (((size_t)(i0 + i) * batch + b) * n_max + r) * d + f0 + e0, o);
            }
        }
        cluster.sync();   // peers have read ss_cta before it is reused or this CTA exits
    }
}

// Many positions (context fill): a persistent grid of one or two CTAs per SM walks the positions
// (no cluster). The T target rows of each position (d contiguous elements each) stream through a ring of
// `ns` shared-memory stages of a few rows as 1-D bulk copies, the stage sequence running on across
// positions. Each stage has a "full" mbarrier (the copies landed) and an "empty" one that every warp
// arrives on once it has read the stage. Thread t forms the D (<= DMAX) draft-layer sums of 8 features or
// (NF 2) two groups of 8 in registers; at the end of a position the D sums of squares take 9 shuffles and one
// named barrier. Every wait is bounded; a CTA that times out sets DFLARE_DEVERR_TIMEOUT and stops.
// Who refills the ring:
// - The warps take turns (PROD false), for many target rows of many features: a warp that only copies would
//   cost every thread a fifth of its registers, and with two feature groups (D 6 to 8: half the reads of the
//   weights alpha per sum, which at one group cost as many shared-memory clocks as the rows) the 128 sums of
//   eight draft layers did not fit beside it.
// - A producer warp (PROD), for few rows or few features: there a position takes a few hundred clocks, the others
//   wait at its barrier for the warp whose turn it is, and a CTA of few warps has registers to spare.
// Bound by HBM for up to four draft layers, by the fp32 FMAs above (10.4k of 20k clocks a position at D 8,
// d 4096). Measured, T 36, target rows read + fused rows written per second, by turns against an earlier form with
// a producer warp, one group and three barriers a position: d 4096 D 8 4.0 -> 4.8 TB/s, D 4 5.5 -> 6.3, D 2
// 5.5 -> 6.2; d 2560 D 5 (2048 positions) 4.3 -> 4.7. Stages of 3 / 4 / 6 / 9 rows at D 8: 679 / 652 / 631 / 827 us
// for 8192 positions; refilling one stage behind instead of two 631 -> 615. 2048 positions (us), the earlier form /
// by turns / with the producer warp: d 1024 D 8 T 8 47 / 67 / 45, d 512 D 6 T 12 56 / 61 / 41, d 256 D 1 T 36
// 40 / 45 / 30, d 4096 D 2 T 4 39 / 43 / 40, fp32 d 512 D 2 T 8 21 / 27 / 21.
constexpr int kLag = 1;         // stages between a slot's use and its refill
constexpr int kMaxNS = 16;      // most stages in the ring
constexpr int kMinNS = 3;
constexpr size_t kRingBytes = 200 * 1024;
constexpr uint64_t kFillWaitNs = 2000000000ull;

__device__ __forceinline__ bool fill_try(uint32_t bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    return done != 0;
}
// Bounded wait; the timer is read only after 64 unsuccessful polls (a %globaltimer read costs a
// few hundred ns, and most waits of the ring complete within those polls).
__device__ __forceinline__ bool fill_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    for (int i = 0; i < 64; ++i)
        if (fill_try(bar, parity)) return true;
    const uint64_t t0 = globaltimer_ns();
    for (int it = 0;; ++it) {
        if (fill_try(bar, parity)) return true;
        if ((it & 63) == 63) {
            if (*abort_flag) return false;
            if (globaltimer_ns() - t0 > kFillWaitNs) {
                *abort_flag = 1;
                return false;
            }
        }
    }
}

// Waits, within one limit for all of them, for the copies of a ring of ns slots whose next stage to read is the one
// in slot st (its full barrier's phase: `phase`). A slot that was not refilled uses the limit up.
__device__ __forceinline__ void fill_drain(uint32_t full_bar0, int ns, int st, uint32_t phase, uint32_t* err) {
    atomicOr(err, DFLARE_DEVERR_TIMEOUT);
    const uint64_t t0 = globaltimer_ns();
    for (int i = 0; i < ns; ++i)
        while (!fill_try(full_bar0 + 8u * i, i >= st ? phase : phase ^ 1u) && globaltimer_ns() - t0 < kFillWaitNs) {
        }
}

// Two fp32 lanes in one 64-bit register: the fill's sums use the paired FMA (fma.rn.f32x2, each
// lane rounded as a scalar fmaf), which halves the instructions of the 8 x D FMAs per row.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pk2(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void upk2(f32x2 v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// 8 consecutive elements of a staged row as four fp32 pairs
__device__ __forceinline__ void load8x2(const bf16* p, f32x2* h) {
    const uint4 u = *reinterpret_cast<const uint4*>(p);
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) h[q] = pk2(__uint_as_float(w[q] << 16), __uint_as_float(w[q] & 0xFFFF0000u));
}
__device__ __forceinline__ void load8x2(const float* p, f32x2* h) {
    const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
    h[0] = pk2(a.x, a.y);
    h[1] = pk2(a.z, a.w);
    h[2] = pk2(b.x, b.y);
    h[3] = pk2(b.z, b.w);
}

// target rows per stage, and up to how many a producer warp refills the ring whatever the features (see fuse_layers_t)
template <class T, bool PROD>
constexpr int kRowsPerStage = sizeof(T) == 2 ? 6 : PROD ? 4 : 3;
template <class T>
constexpr int kFewRows = sizeof(T) == 2 ? 8 : 4;

template <class T, int DMAX, int NF, bool PROD>
__device__ __forceinline__ void fuse_rows_body(
    const T* __restrict__ H, const float* __restrict__ alpha, const T* __restrict__ gain,
    T* __restrict__ F, T* __restrict__ F_out, const int32_t* __restrict__ app_cnt, int D, int Tn,
    int batch, int n_max, int d, long long f_layer_rows, float eps, int ns, uint32_t* err) {
    constexpr int kRB = kRowsPerStage<T, PROD>;
    pdl_trigger();
    extern __shared__ __align__(128) uint8_t stage_mem[];   // [ns][kRB][d]
    constexpr int DP = (DMAX + 1) & ~1;                       // DMAX rounded up to even
    __shared__ __align__(16) f32x2 s_alpha[64 * DP];          // [j][i] = (alpha_ij, alpha_ij), Tn <= 64
    __shared__ float red[2][16][8];       // the warps' sums of squares, by parity of the position
    __shared__ int s_cnt[64];             // appended rows per sequence
    __shared__ __align__(8) uint64_t full_bar[kMaxNS], empty_bar[kMaxNS];
    __shared__ int abort_flag;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_cw = (int)(blockDim.x >> 5) - (PROD ? 1 : 0), n_ct = PROD ? n_cw * 32 : (int)blockDim.x;   // that form sums
    const uint32_t fb0 = (uint32_t)__cvta_generic_to_shared(&full_bar[0]);
    const uint32_t eb0 = (uint32_t)__cvta_generic_to_shared(&empty_bar[0]);
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(stage_mem);
    if (tid == 0) {
        for (int i = 0; i < ns; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(fb0 + 8u * i) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(eb0 + 8u * i), "r"(n_cw) : "memory");
        }
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    pdl_wait();
    for (int k = tid; k < Tn * DP; k += blockDim.x) {
        const int j = k / DP, i = k % DP;
        const float a = i < D ? alpha[i * Tn + j] : 0.f;
        s_alpha[k] = pk2(a, a);
    }
    for (int k = tid; k < batch; k += blockDim.x) s_cnt[k] = app_cnt[k];
    __syncthreads();
    volatile int* abrt = &abort_flag;
    const int n_pos = batch * n_max;
    const size_t lstride = (size_t)n_pos * d;
    const uint32_t row_bytes = (uint32_t)(d * sizeof(T));
    const int nst = (Tn + kRB - 1) / kRB;   // stages per position
    // this CTA's positions pid = blockIdx.x + k * gridDim.x that have rows to append
    auto valid = [&](int pid) { return pid % n_max < s_cnt[pid / n_max]; };
    auto next_pos = [&](int pid) {
        for (pid += gridDim.x; pid < n_pos; pid += gridDim.x)
            if (valid(pid)) return pid;
        return n_pos;
    };
    int first = (int)blockIdx.x;
    if (first < n_pos && !valid(first)) first = next_pos(first);

    // The stages run on across positions. Stage g goes into slot g % ns. By turns: the ring is filled once at the
    // start, then each step's refill is issued by one elected thread, warp g % n_cw at its step g, into
    // the slot of stage g - kLag, which the other warps have left by then as a rule. (ppid, pk): the
    // next stage to issue, tracked by every thread.
    int ppid = first, pk = 0;
    auto next_stage = [&] {
        if (++pk == nst) {
            pk = 0;
            ppid = next_pos(ppid);
        }
    };
    auto issue = [&](int slot) {
        const int j0 = pk * kRB, nr = min(kRB, Tn - j0);
        const uint32_t bar = fb0 + 8u * slot;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"((uint32_t)nr * row_bytes)
                     : "memory");
        for (int u = 0; u < nr; ++u)
            asm volatile(
                "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                    sbase + (uint32_t)(slot * kRB + u) * row_bytes),
                "l"(H + (size_t)(j0 + u) * lstride + (size_t)ppid * d), "r"(row_bytes), "r"(bar)
                : "memory");
    };
    if constexpr (!PROD)
        for (int i = 0; i < ns && ppid < n_pos; ++i, next_stage())
            if (warp == 0 && elect_one()) issue(i);

    if (PROD && warp == n_cw) {
        if (elect_one()) {
            int st = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (; ppid < n_pos; next_stage()) {
                if (!fill_wait(eb0 + 8u * st, phase ^ 1u, abrt)) {
                    ok = false;
                    break;
                }
                issue(st);
                if (++st == ns) {
                    st = 0;
                    phase ^= 1u;
                }
            }
            // after a timeout: the last copies of every slot land before the CTA leaves
            if (!ok) fill_drain(fb0, ns, st, phase ^ 1u, err);
        }
    } else {
        // thread t owns NF groups of 8 features, n_ct groups apart; a thread without its last group reads
        // group 0 instead and drops the result
        int e[NF], er[NF];
#pragma unroll
        for (int c = 0; c < NF; ++c) {
            e[c] = (tid + c * n_ct) * 8;
            er[c] = e[c] < d ? e[c] : 0;
        }
        const T* stg = reinterpret_cast<const T*>(stage_mem);
        int st = 0, par = 0, turn = 0;         // slot; parity of the position; warp that refills
        int rst = -kLag;                       // slot to refill (negative: none yet)
        uint32_t phase = 0, rphase = 0;
        bool ok = true;
        int bad = 0;
        f32x2 acc2[DMAX][4 * NF];
        // one target row, in G of the NF groups: a warp whose last group lies past d leaves it out
        const bool all_groups = NF == 1 || (warp * 32 + (NF - 1) * n_ct) * 8 < d;
        auto add_row = [&](auto groups, const T* row, int j) {
            constexpr int G = decltype(groups)::value;
            f32x2 h[4 * G];
#pragma unroll
            for (int c = 0; c < G; ++c) load8x2(row + er[c], h + 4 * c);
#pragma unroll
            for (int i = 0; i < DP; i += 2) {
                const uint4 a4 = *reinterpret_cast<const uint4*>(&s_alpha[j * DP + i]);
                const f32x2 a0 = ((f32x2)a4.y << 32) | a4.x, a1 = ((f32x2)a4.w << 32) | a4.z;
#pragma unroll
                for (int q = 0; q < 4 * G; ++q) acc2[i][q] = fma2(a0, h[q], acc2[i][q]);
                if (i + 1 < DMAX) {
                    const int i1 = i + 1 < DMAX ? i + 1 : i;
#pragma unroll
                    for (int q = 0; q < 4 * G; ++q) acc2[i1][q] = fma2(a1, h[q], acc2[i1][q]);
                }
            }
        };
        for (int pid = first; pid < n_pos; pid = next_pos(pid)) {
            const int b = pid / n_max, r = pid % n_max;
#pragma unroll
            for (int i = 0; i < DMAX; ++i)
#pragma unroll
                for (int q = 0; q < 4 * NF; ++q) acc2[i][q] = 0ull;
            for (int k = 0; k < nst; ++k) {
                if (!__all_sync(0xffffffffu, fill_wait(fb0 + 8u * st, phase, abrt))) {
                    ok = false;
                    break;
                }
                const T* row = stg + (size_t)st * kRB * d;
                auto add_stage = [&](auto groups) {
                    if ((k + 1) * kRB <= Tn) {   // no branch between the rows: their loads are in flight together
#pragma unroll
                        for (int u = 0; u < kRB; ++u) add_row(groups, row + u * d, k * kRB + u);
                    } else {
                        for (int j = k * kRB; j < Tn; ++j, row += d) add_row(groups, row, j);
                    }
                };
                if (all_groups)
                    add_stage(std::integral_constant<int, NF>{});
                else if constexpr (NF > 1)
                    add_stage(std::integral_constant<int, NF - 1>{});
                __syncwarp();
                if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(eb0 + 8u * st) : "memory");
                if (!PROD && rst >= 0 && ppid < n_pos) {
                    if (warp == turn && elect_one()) {
                        if (fill_wait(eb0 + 8u * rst, rphase, abrt))
                            issue(rst);
                        else
                            ok = false;
                    }
                    next_stage();
                }
                if (++turn == n_cw) turn = 0;
                if (++rst == ns) {
                    rst = 0;
                    rphase ^= 1u;
                }
                if (++st == ns) {
                    st = 0;
                    phase ^= 1u;
                }
            }
            // the first gains of bf16 rows arrive behind the reduction, the others kGP layers ahead
            constexpr int kGP = DMAX < 4 ? DMAX : 4;
            uint4 graw[kGP][NF];
            auto fetch_gain = [&](int i) {
                if constexpr (sizeof(T) == 2) {
                    if (i < D) {
#pragma unroll
                        for (int c = 0; c < NF; ++c)
                            graw[i % kGP][c] = __ldg(reinterpret_cast<const uint4*>(gain + (size_t)i * d + er[c]));
                    }
                }
            };
#pragma unroll
            for (int i = 0; i < kGP; ++i) fetch_gain(i);
            // sums of squares: eight values over 32 lanes by halving exchanges (9 shuffles; lane holds
            // value lane / 4 at the end), the warps' sums through shared memory
            float v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = 0.f;
#pragma unroll
            for (int i = 0; i < DMAX; ++i) {
#pragma unroll
                for (int c = 0; c < NF; ++c) {
                    f32x2 s2 = 0ull;
#pragma unroll
                    for (int q = 0; q < 4; ++q) s2 = fma2(acc2[i][4 * c + q], acc2[i][4 * c + q], s2);
                    float lo, hi;
                    upk2(s2, lo, hi);
                    if (e[c] < d) v[i] += lo + hi;
                }
            }
#pragma unroll
            for (int n = 4, o = 16; n > 0; n >>= 1, o >>= 1) {
                const bool up = lane & o;
#pragma unroll
                for (int i = 0; i < n; ++i) {
                    const float give = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
                    v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
                }
            }
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
            if ((lane & 3) == 0) red[par][warp][lane >> 2] = v[0];
            // one barrier a position: it also tells every consumer whether one of them timed out, so
            // that they leave together
            asm volatile(
                "{\n\t.reg .pred p, q;\n\t"
                "setp.ne.s32 p, %1, 0;\n\t"
                "barrier.cta.red.or.pred q, 1, %2, p;\n\t"
                "selp.s32 %0, 1, 0, q;\n\t}"
                : "=r"(bad)
                : "r"(ok ? 0 : 1), "r"(n_ct)
                : "memory");
            if (bad) break;
            // every warp adds the warps' sums itself: lane = value lane % 8, warps lane / 8, + 4, ...
            float tot = 0.f;
            for (int w = lane >> 3; w < n_cw; w += 4) tot += red[par][w][lane & 7];
            tot += __shfl_xor_sync(0xffffffffu, tot, 8);
            tot += __shfl_xor_sync(0xffffffffu, tot, 16);
            const float inv_l = inv_rms(tot, d, eps);
            par ^= 1;
#pragma unroll
            for (int i = 0; i < DMAX; ++i) {
                if (i >= D) break;
                const float inv = __shfl_sync(0xffffffffu, inv_l, i);
#pragma unroll
                for (int c = 0; c < NF; ++c) {
                    if (e[c] >= d) continue;
                    float gg[8], o[8];
                    if constexpr (sizeof(T) == 2)
                        load8(reinterpret_cast<const T*>(&graw[i % kGP][c]), gg);
                    else
                        load8(gain + (size_t)i * d + e[c], gg);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        float lo, hi;
                        upk2(acc2[i][4 * c + q], lo, hi);
                        o[2 * q] = gg[2 * q] * (lo * inv);
                        o[2 * q + 1] = gg[2 * q + 1] * (hi * inv);
                    }
                    store8(F + ((size_t)i * f_layer_rows + pid) * d + e[c], o);
                    if (F_out) store8(F_out + (((size_t)i * batch + b) * n_max + r) * d + e[c], o);
                }
                if (i + kGP < DMAX) fetch_gain(i + kGP);
            }
        }
        // after a timeout: the copies in flight, none beyond the stage that this thread reads next from their
        // slot, land before the CTA leaves, within one more limit for all slots
        if (bad && tid == 0) fill_drain(fb0, ns, st, phase, err);
    }
    __syncthreads();
}

#define FUSE_ROWS_PARAMS                                                                            \
    const T *__restrict__ H, const float *__restrict__ alpha, const T *__restrict__ gain,           \
        T *__restrict__ F, T *__restrict__ F_out, const int32_t *__restrict__ app_cnt, int D,         \
        int Tn, int batch, int n_max, int d, long long f_layer_rows, float eps, int ns, uint32_t *err
#define FUSE_ROWS_ARGS H, alpha, gain, F, F_out, app_cnt, D, Tn, batch, n_max, d, f_layer_rows, eps, ns, err
template <class T, int DMAX, int NF>
__global__ void __launch_bounds__(512 / NF, 1) fuse_rows_kernel(FUSE_ROWS_PARAMS) {
    fuse_rows_body<T, DMAX, NF, false>(FUSE_ROWS_ARGS);
}
template <class T, int DMAX>
__global__ void __launch_bounds__(320, 2) fuse_rows2_kernel(FUSE_ROWS_PARAMS) {
    fuse_rows_body<T, DMAX, 1, false>(FUSE_ROWS_ARGS);
}
template <class T, int DMAX, int THREADS, int PER_SM>
__global__ void __launch_bounds__(THREADS + 32, PER_SM) fuse_rows_prod_kernel(FUSE_ROWS_PARAMS) {
    fuse_rows_body<T, DMAX, 1, true>(FUSE_ROWS_ARGS);
}
#undef FUSE_ROWS_PARAMS
#undef FUSE_ROWS_ARGS

template <class T>
cudaError_t fuse_layers_t(dflare_ctx* c, const void* hidden, int n_max, void* fused_out,
                          cudaStream_t s) {
    const dflare_config& g = c->cfg;
    const int C = (g.d + kFuseCH - 1) / kFuseCH;
    const size_t smem = (size_t)(g.n_target_layers + g.n_draft_layers) * kFuseCH * sizeof(T) +
                        (size_t)(kFuseGroups - 1) * 8 * 8 * 64 * sizeof(float);
    const T* H = static_cast<const T*>(hidden);
    const T* gain = static_cast<const T*>(c->w.fuse_norm);
    T* F = static_cast<T*>(c->fused);
    T* Fo = static_cast<T*>(fused_out);
    // Context fill: CTAs of d / 8 threads, or of d / 16 where six to eight draft layers take two feature groups per
    // thread, two per SM when their registers allow (rings of about 100 KB), else one (about 200 KB); at most kMaxNS
    // stages. A producer warp refills the ring up to 1024 features, or 2560 at six to eight draft layers (where its
    // CTA has registers for one group's sums), and for up to kFewRows target rows, unless two CTAs fit on an SM only
    // without it. Across those lines, 2048 positions, by turns / producer warp (us): d 1024 D 4 T 36 45.2 / 42.9, d 1536
    // D 2 T 24 10 % behind with the producer warp, d 2048 D 4 T 8 33.6 / 31.6, d 2048 D 6 T 36 121.7 / 102.4, fp32 d 1024
    // D 2 T 12 31.6 / 31.6; d 2560 D 8 T 36 1.19 times by turns. (Six to eight draft layers of more features
    // stay by turns: the producer's CTA would spill.)
    const int Dn = g.n_draft_layers, nf = Dn <= 5 ? 1 : 2, d_threads = (g.d / 8 + 31) / 32 * 32;   // (d <= 4096)
    const size_t prod_stage = (size_t)kRowsPerStage<T, true> * g.d * sizeof(T);
    const bool two_prod = d_threads <= (Dn <= 2 ? 320 : 256) && kMinNS * prod_stage <= kRingBytes / 2;
    const bool few = g.n_target_layers <= kFewRows<T> && (two_prod || (Dn < 5 && d_threads > 320));
    const bool prod = Dn > 5 ? d_threads <= 320 : g.d <= 1024 || few;
    const size_t stage_bytes = prod ? prod_stage : (size_t)kRowsPerStage<T, false> * g.d * sizeof(T);
    if ((long long)c->batch * n_max >= 2LL * c->num_sms && Dn <= 8 && g.n_target_layers <= 64 &&
        kMinNS * stage_bytes <= kRingBytes) {
        // each variant is set up, and with that loaded, when it is first taken: all nine at once moved what a program
        // allocates after its first fill, and with it other launches (Qwen3-4B block 402.5 -> 407.2 us)
        enum { BY_TURNS_4, BY_TURNS_5, BY_TURNS_8, TWO_BY_TURNS_4, TWO_BY_TURNS_5, PROD_4, TWO_PROD_2, TWO_PROD_5, PROD_8, VARIANTS };
        using Fill = decltype(&fuse_rows_kernel<T, 4, 1>);
        static const Fill variant[VARIANTS] = {
            fuse_rows_kernel<T, 4, 1>, fuse_rows_kernel<T, 5, 1>, fuse_rows_kernel<T, 8, 2>, fuse_rows2_kernel<T, 4>,
            fuse_rows2_kernel<T, 5>, fuse_rows_prod_kernel<T, 4, 512, 1>, fuse_rows_prod_kernel<T, 2, 320, 2>,
            fuse_rows_prod_kernel<T, 5, 256, 2>, fuse_rows_prod_kernel<T, 8, 320, 1>};
        static PerDeviceOnce ready[VARIANTS];
        auto set_up = [](int i) {
            return ready[i]([i] {
                return cudaFuncSetAttribute(variant[i], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRingBytes);
            });
        };
        // v2: two CTAs per SM, where they fit; v: one (with a producer warp the same kernel, if it has one for two)
        const int v2 = prod ? (d_threads <= 256 ? TWO_PROD_5 : TWO_PROD_2) : Dn <= 4 ? TWO_BY_TURNS_4 : TWO_BY_TURNS_5;
        int v = prod ? (Dn > 5 ? PROD_8 : d_threads <= 320 ? v2 : PROD_4)
                     : Dn <= 4 ? BY_TURNS_4 : Dn == 5 ? BY_TURNS_5 : BY_TURNS_8;
        int ns = (int)std::min<size_t>(kMaxNS, kRingBytes / stage_bytes), per_sm = 1;
        const int ns2 = (int)std::min<size_t>(kMaxNS, kRingBytes / 2 / stage_bytes);
        const int threads = prod ? d_threads + 32 : std::min(512 / nf, d_threads);
        if (Dn <= 5 && ns2 >= kMinNS && d_threads <= 320) {
            int fit = 0;
            if (set_up(v2) == cudaSuccess &&
                cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, variant[v2], threads, (size_t)ns2 * stage_bytes) ==
                    cudaSuccess && fit >= 2) {
                v = v2;
                ns = ns2;
                per_sm = 2;
            }
        }
        const cudaError_t re = set_up(v);
        if (re != cudaSuccess) return re;
        const int grid = (int)std::min<long long>((long long)c->batch * n_max, (long long)per_sm * c->num_sms);
        return launch_kernel(c->pdl, variant[v], dim3(grid), dim3(threads), (size_t)ns * stage_bytes, s, H,
                             (const float*)c->alpha, gain, F, Fo, (const int32_t*)c->app_cnt,
                             g.n_draft_layers, g.n_target_layers, c->batch, n_max, g.d,
                             (long long)g.max_fuse_rows, g.rms_eps, ns, c->err);
    }
    auto kern = g.n_draft_layers <= 4 ? fuse_layers_kernel<T, 4> : fuse_layers_kernel<T, 8>;
    static PerDeviceOnce configured;
    const cudaError_t ce = configured([] {
        for (auto k : {fuse_layers_kernel<T, 4>, fuse_layers_kernel<T, 8>}) {
            cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)((64 + 16) * kFuseCH * sizeof(T) +
                                                       (kFuseGroups - 1) * 8 * 8 * 64 * 4));
            if (e != cudaSuccess) return e;
        }
        return cudaSuccess;
    });
    if (ce != cudaSuccess) return ce;
    return launch_cluster(c->pdl, C, kern, dim3(C, n_max, c->batch), dim3(256), smem, s, H,
                          (const float*)c->alpha, gain, F, Fo, (const int32_t*)c->app_cnt,
                          g.n_draft_layers, g.n_target_layers, c->batch, n_max, g.d,
                          (long long)g.max_fuse_rows, g.rms_eps);
}

}  // namespace

cudaError_t launch_fusion_alpha(dflare_ctx* c, cudaStream_t s) {
    const dflare_config& g = c->cfg;
    return launch_kernel(c->pdl, fusion_alpha_kernel, dim3(1),
                         dim3(32 * ((g.n_draft_layers + 31) / 32)), 0, s,
                         (const float*)c->w.fuse_logits, c->alpha, g.n_draft_layers,
                         g.n_target_layers, (g.flags & DFLARE_FLAG_RAW_FUSION) ? 1 : 0);
}

cudaError_t launch_fuse_begin(dflare_ctx* c, const int32_t* n_new, int n_max, cudaStream_t s) {
    return launch_kernel(c->pdl, fuse_begin_kernel, dim3(1), dim3(64), 0, s, c->ctx_len,
                         c->app_base, c->app_cnt, n_new, c->batch, n_max, c->cfg.max_ctx, c->err);
}

cudaError_t launch_fuse_layers(dflare_ctx* c, const void* hidden, int n_max, void* fused_out,
                               cudaStream_t s) {
    if (c->cfg.dtype == DFLARE_F32) return fuse_layers_t<float>(c, hidden, n_max, fused_out, s);
    return fuse_layers_t<bf16>(c, hidden, n_max, fused_out, s);
}

}  // namespace dfl
