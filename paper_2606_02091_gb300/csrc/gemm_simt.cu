// CUDA-core projection GEMM: the fp32 storage mode's GEMM (exact fp32 products, which the
// tensor cores do not offer) and, for bf16, a diagnostic cross-check of the tcgen05 GEMM.
//
// The fp32 drafters are small (hidden size of a few hundred, a handful of token rows), so a
// projection is bound by the latency of its longest chain, not by bandwidth. One CTA takes 32
// weight rows x TT tokens over the whole K range, one warp four rows: a lane holds 4 consecutive k
// of every 128, multiplies them with the same k of all TT tokens (64 sums in registers at 16
// tokens), and the 32 lanes' sums are added in a butterfly that halves the values a lane holds at
// each step. No shared memory and no barrier until the epilogue, the first weights are loaded
// before the dependency wait, and a lane's serial chain is K / 32 FMAs per sum. Each 16-byte load
// feeds 16 (weights: 4 TT) FMAs; projections of many token rows take the tiled form below. The
// earlier form (128 rows x 16 tokens per CTA, K in shared-memory chunks of 16 between
// two barriers) waited a memory round trip per chunk (ncu: 32 us at K 256, 92 us at K 768). With this
// kernel and the fp32 attention of attention.cu the first step of a 128-position sequence on the fp32
// drafter (d 256, 4 layers, block 8) went from 968 to 158 us, and to 134 with two chunks of K per round.
#include "epilogue.cuh"

#include <algorithm>

namespace dfl {
namespace {

constexpr int kRows = 32;      // weight rows per CTA: two groups of 16 features (SwiGLU: one group
                               // of gate and the same 16 features of up)
constexpr int kSimtThreads = 256;

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 ld4(const bf16* p) {
    const uint2 u = *reinterpret_cast<const uint2*>(p);
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u),
                       __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xFFFF0000u));
}

// TT: tokens per CTA (8 or 16). blockIdx.x = group * n_slices + slice, blockIdx.y = token chunk.
template <class T, int TT>
__global__ void __launch_bounds__(kSimtThreads) gemm_simt_kernel(
    const T* __restrict__ A, const T* __restrict__ A2, const T* __restrict__ Bm, int n, int k, int m_tok,
    long long a_group_rows, long long b_group_rows, int b_shared, int b_kgroup, int n_slices, EpiParams ep) {
    __shared__ __align__(16) float tile[2 * kEpiChunk * 128];   // the epilogue's [acc][token][feature]
    const int slice = blockIdx.x % n_slices, group = blockIdx.x / n_slices;
    const int tok0 = blockIdx.y * TT;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // the CTA's two groups of 16 features; a projection with a rotary epilogue takes a group and its
    // rotary partner half a head further, so that the epilogue finds both in its tile
    int f_a, f_b;
    if (A2) {
        f_a = f_b = slice * 16;
    } else if (ep.kind == EPI_QKV || ep.kind == EPI_KV_APPEND) {
        const int q = slice & 3;
        f_a = (slice >> 2) * 128 + (ep.head_dim == 64 ? (q >> 1) * 64 + (q & 1) * 16 : q * 16);
        f_b = f_a + (ep.head_dim >> 1);
    } else {
        f_a = slice * 32;
        f_b = f_a + 16;
    }
    const int sub = (warp & 3) * 4;                     // the warp's first row within its group
    const int row0 = (warp < 4 ? f_a : f_b) + sub;
    const T* Ag = (A2 && warp >= 4 ? A2 : A) + (size_t)group * a_group_rows * k;
    const T* wp[4];
#pragma unroll
    for (int f = 0; f < 4; ++f) wp[f] = Ag + (size_t)min(row0 + f, n - 1) * k + 4 * lane;   // rows past n: not stored
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    // KC chunks of 128 k per round, whose loads are in flight together: the fp32 step above 158 us with one,
    // 134 with two, 139 with three (254 registers: the next launch starts later; at 16 tokens a second
    // chunk would spill)
    constexpr int KC = TT == 8 ? 2 : 1;
    float4 w[KC][4];
#pragma unroll
    for (int j = 0; j < KC; ++j)
#pragma unroll
        for (int f = 0; f < 4; ++f) w[j][f] = 4 * lane + 128 * j < k ? ld4(wp[f] + 128 * j) : zero;
    pdl_wait();
    pdl_trigger();   // after the wait: see gemm_tc_kernel
    const T* Bg = Bm + (size_t)(b_shared || b_kgroup > 0 ? 0 : group) * b_group_rows * k;
    const size_t b_ld = b_kgroup > 0 ? b_kgroup : k;    // elements between token rows
    float acc[4 * TT];
#pragma unroll
    for (int i = 0; i < 4 * TT; ++i) acc[i] = 0.f;
    for (int c0 = 0; c0 < k; c0 += 128 * KC) {
        float4 x[KC][TT];
#pragma unroll
        for (int j = 0; j < KC; ++j) {
            const int col = c0 + 128 * j + 4 * lane;
            const bool in = col < k;
            const T* bp = Bg + col;
            if (b_kgroup > 0) {   // contraction over stacked activation groups (Eq. 1)
                const int z = col / b_kgroup;
                bp = Bm + (size_t)z * b_group_rows * b_kgroup + (col - z * b_kgroup);
            }
#pragma unroll
            for (int t = 0; t < TT; ++t) x[j][t] = in ? ld4(bp + (size_t)min(tok0 + t, m_tok - 1) * b_ld) : zero;
        }
#pragma unroll
        for (int j = 0; j < KC; ++j) {
            float4 wn[4];
            const int next = c0 + 128 * (KC + j);
#pragma unroll
            for (int f = 0; f < 4; ++f) wn[f] = next + 4 * lane < k ? ld4(wp[f] + next) : zero;
#pragma unroll
            for (int f = 0; f < 4; ++f)
#pragma unroll
                for (int t = 0; t < TT; ++t) {
                    float a = acc[f * TT + t];
                    a = fmaf(w[j][f].x, x[j][t].x, a);
                    a = fmaf(w[j][f].y, x[j][t].y, a);
                    a = fmaf(w[j][f].z, x[j][t].z, a);
                    acc[f * TT + t] = fmaf(w[j][f].w, x[j][t].w, a);
                }
#pragma unroll
            for (int f = 0; f < 4; ++f) w[j][f] = wn[f];
        }
    }
    // add the 32 lanes' sums: at each step a lane keeps one half of its values (the upper half when
    // its lane bit is set) and gives the other away; afterwards it holds values 4 TT / 32 * lane ..
    constexpr int kLeft = 4 * TT / 32;
#pragma unroll
    for (int o = 16, half = 2 * TT; o > 0; o >>= 1, half >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const float give = up ? acc[i] : acc[i + half];
            const float keep = up ? acc[i + half] : acc[i];
            acc[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    float* const dst = tile + (A2 && warp >= 4 ? kEpiChunk * 128 : 0) + (row0 & 127);
#pragma unroll
    for (int i = 0; i < kLeft; ++i) {
        const int v = lane * kLeft + i;                 // value f * TT + t
        dst[(v % TT) * 128 + v / TT] = acc[i];
    }
    __syncthreads();
    const int c = threadIdx.x >> 1, g = threadIdx.x & 1;
    if (c < TT && !(A2 && g)) {
        const int f0 = g ? f_b : f_a;
        apply_epilogue<T>(ep, tile, group, f0 >> 7, tok0, c * 8 + ((f0 & 127) >> 4));
    }
}

// Many token rows, or a short K under many weight rows: one CTA computes 128 weight rows x TOK tokens (SwiGLU: 128 of
// gate, the same 128 of up x 32 tokens), TOK 64 as 8 x 4 sums per thread (2 x 8 x 2), TOK 16 as 8 x 1, K in chunks of
// 16 through two shared-memory buffers, the next chunk's loads in flight behind the FMAs. Bound by the FMAs and the
// shared-memory reads that feed them. The warp-per-rows form, whose eight warps each load the tokens for themselves
// and pay its butterfly and its rounds of 128 k whatever K is, had fallen behind the one before it here (us, the one
// before / warp per rows / tiles): K 1024, 16384 rows x 512 1180 / 1389 / 508; K 512, 32768 x 512 1174 / 1522 / 535; K 256,
// 8192 x 256 97 / 106 / 47; K 64, 151936 features, 15 rows 31 / 65 / 33 (TOK 16), 60 rows 98 / 246 / 61; K 192, 151936
// features, 15 rows 84 / 105 / 82. What is left behind: 151936 features at K 64 and 128, up to 30 rows, 4 to 15 %.
// A thread adds a chunk's products in four chains of 4, which are added pairwise. TREE: chunks are added pairwise too,
// and each four of them to the total (K up to 128, at 20 % more time than without); otherwise four in a row and that to the
// total. The error against 64 bits is then no larger than the warp-per-rows form's (rms, of the result's, in 1e-8;
// warp per rows / tree / no tree): K 64 6.77 / 6.77 / 6.90, K 128 7.29 / 7.29 / 7.41, K 192 7.85 / - / 7.74, K 256
// 8.14 / - / 8.01, K 2048 15.7 / - / 12.7. (Chains of 8 would save 5 % and have 7.77 at K 128 and 8.33 at K 256.)
constexpr int kTileK = 16, kChain = 4;
template <class T, bool DUAL, int TOK, bool TREE>
__global__ void __launch_bounds__(kSimtThreads, TOK == 16 ? 2 : 1) gemm_simt_tiled_kernel(
    const T* __restrict__ A, const T* __restrict__ A2, const T* __restrict__ Bm, int n, int k, int m_tok,
    long long a_group_rows, long long b_group_rows, int b_shared, int b_kgroup, int n_tiles, EpiParams ep) {
    constexpr int NA = DUAL ? 2 : 1, TPT = TOK / 16;   // accumulators, tokens per thread
    constexpr int LDA = 128 + 4, LDB = TOK + 4;
    constexpr int OPS = 2 * kTileK * (NA * LDA + LDB), TILES = NA * TOK * 128;
    __shared__ __align__(16) float buf[OPS > TILES ? OPS : TILES];   // operands, then the epilogue's tiles
    const int n_tile = blockIdx.x % n_tiles, group = blockIdx.x / n_tiles, tok0 = blockIdx.y * TOK;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const T* Bg = Bm + (size_t)(b_shared || b_kgroup > 0 ? 0 : group) * b_group_rows * k;
    const size_t b_ld = b_kgroup > 0 ? b_kgroup : k;
    const int lr = tid >> 2, lk = (tid & 3) * 4;    // this thread's row (+ 64) and k of a chunk's loads
    const T* ap[NA][2];
#pragma unroll
    for (int a = 0; a < NA; ++a)
#pragma unroll
        for (int h = 0; h < 2; ++h)
            ap[a][h] = (a ? A2 : A) + ((size_t)group * a_group_rows + min(n_tile * 128 + lr + 64 * h, n - 1)) * k + lk;
    const bool lb = lr < TOK;
    const T* const bp = Bg + (size_t)min(tok0 + (lb ? lr : 0), m_tok - 1) * b_ld + lk;   // rows past the end: not stored
    auto b_at = [&](int k0) {   // contraction over stacked activation groups (Eq. 1): a chunk lies in one
        if (b_kgroup <= 0) return bp + k0;
        const int z = k0 / b_kgroup;
        return bp + (size_t)z * b_group_rows * b_kgroup + (k0 - z * b_kgroup);
    };
    auto As = [&](int st, int a) { return buf + (st * NA + a) * kTileK * LDA; };
    auto Bs = [&](int st) { return buf + 2 * NA * kTileK * LDA + st * kTileK * LDB; };
    float4 ra[NA][2], rb = make_float4(0.f, 0.f, 0.f, 0.f);
    auto load_a = [&](int k0) {
#pragma unroll
        for (int a = 0; a < NA; ++a)
#pragma unroll
            for (int h = 0; h < 2; ++h) ra[a][h] = ld4(ap[a][h] + k0);
    };
    auto load_b = [&](int k0) {
        if (lb) rb = ld4(b_at(k0));
    };
    auto put = [&](float* d, int ld, float4 v) {
        d[0] = v.x;
        d[ld] = v.y;
        d[2 * ld] = v.z;
        d[3 * ld] = v.w;
    };
    auto store = [&](int st) {
#pragma unroll
        for (int a = 0; a < NA; ++a)
#pragma unroll
            for (int h = 0; h < 2; ++h) put(As(st, a) + lk * LDA + lr + 64 * h, LDA, ra[a][h]);
        if (lb) put(Bs(st) + lk * LDB + lr, LDB, rb);
    };
    constexpr int S = NA * 8 * TPT;                 // sums of a thread, [accumulator][feature][token]
    float acc[S], part[S], pair[S];
#pragma unroll
    for (int i = 0; i < S; ++i) acc[i] = part[i] = 0.f;
    load_a(0);
    pdl_wait();
    pdl_trigger();   // after the wait: see gemm_tc_kernel
    load_b(0);
    store(0);
    __syncthreads();
    const int chunks = k / kTileK;   // (k is a multiple of 64)
    for (int c = 0; c < chunks; ++c) {
        const int st = c & 1;
        if (c + 1 < chunks) {
            load_a((c + 1) * kTileK);
            load_b((c + 1) * kTileK);
        }
        constexpr int NC = kTileK / kChain;
        float sum[NC][S];
#pragma unroll
        for (int h = 0; h < NC; ++h) {
#pragma unroll
            for (int i = 0; i < S; ++i) sum[h][i] = 0.f;
#pragma unroll
            for (int kk = h * kChain; kk < (h + 1) * kChain; ++kk) {
                float b[TPT];
#pragma unroll
                for (int t = 0; t < TPT; ++t) b[t] = Bs(st)[kk * LDB + ty * TPT + t];
#pragma unroll
                for (int a = 0; a < NA; ++a) {
                    const float4 lo = *reinterpret_cast<const float4*>(As(st, a) + kk * LDA + tx * 4);
                    const float4 hi = *reinterpret_cast<const float4*>(As(st, a) + kk * LDA + 64 + tx * 4);
                    const float w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
                    for (int f = 0; f < 8; ++f)
#pragma unroll
                        for (int t = 0; t < TPT; ++t) {
                            float& x = sum[h][(a * 8 + f) * TPT + t];
                            x = fmaf(w[f], b[t], x);
                        }
                }
            }
        }
#pragma unroll
        for (int i = 0; i < S; ++i) sum[0][i] = (sum[0][i] + sum[1][i]) + (sum[2][i] + sum[3][i]);
        if (TREE) {
            if (!(c & 1)) {
#pragma unroll
                for (int i = 0; i < S; ++i) pair[i] = sum[0][i];
            } else {
#pragma unroll
                for (int i = 0; i < S; ++i) pair[i] += sum[0][i];
                if (!(c & 2)) {
#pragma unroll
                    for (int i = 0; i < S; ++i) part[i] = pair[i];
                } else {
#pragma unroll
                    for (int i = 0; i < S; ++i) acc[i] += part[i] + pair[i];
                }
            }
        } else {
#pragma unroll
            for (int i = 0; i < S; ++i) part[i] += sum[0][i];
            if ((c & 3) == 3) {
#pragma unroll
                for (int i = 0; i < S; ++i) {
                    acc[i] += part[i];
                    part[i] = 0.f;
                }
            }
        }
        if (c + 1 < chunks) store(st ^ 1);   // (read two chunks ago, before the last barrier)
        __syncthreads();
    }
    // the epilogue's tiles [16-token chunk][accumulator][token][feature]
#pragma unroll
    for (int a = 0; a < NA; ++a)
#pragma unroll
        for (int t = 0; t < TPT; ++t) {
            const int tok = ty * TPT + t;
            float* d = buf + (((tok >> 4) * NA + a) * kEpiChunk + (tok & 15)) * 128 + tx * 4;
            const float* v = acc + a * 8 * TPT + t;
            *reinterpret_cast<float4*>(d) = make_float4(v[0], v[TPT], v[2 * TPT], v[3 * TPT]);
            *reinterpret_cast<float4*>(d + 64) = make_float4(v[4 * TPT], v[5 * TPT], v[6 * TPT], v[7 * TPT]);
        }
    __syncthreads();
    for (int ch = tid >> 7; ch < TOK / kEpiChunk; ch += 2)
        apply_epilogue<T>(ep, buf + ch * NA * kEpiChunk * 128, group, n_tile, tok0 + ch * kEpiChunk, tid & 127);
}

template <class T>
cudaError_t launch_t(dflare_ctx* c, const GemmDesc& g, cudaStream_t s) {
    const long long a_gr = g.a_group_rows > 0 ? g.a_group_rows : g.n;
    const int per = g.a2 ? 16 : kRows, n_slices = (g.n + per - 1) / per, tt = g.m_tok <= 8 ? 8 : 16;
    const long long warp_ctas = (long long)n_slices * g.groups * ((g.m_tok + tt - 1) / tt);
    const int n_tiles = (g.n + 127) / 128;
    auto tiled = [&](auto kernel, int tok) {
        return launch_kernel(c->pdl, kernel, dim3(n_tiles * g.groups, (g.m_tok + tok - 1) / tok), dim3(kSimtThreads), 0, s,
                             (const T*)g.a, (const T*)g.a2, (const T*)g.b, g.n, g.k, g.m_tok, a_gr, g.b_group_rows,
                             g.b_shared, g.b_kgroup, n_tiles, g.ep);
    };
    // A wave of tiles, one per SM, takes as long as about ten CTAs per SM of the warp-per-rows form (SwiGLU: eleven), and
    // as six where K is short, which that form pays by 128 (SwiGLU at K 64: four). Measured, warp-per-rows / tiles (us):
    // K 64, 120 rows x 8192 (13 CTAs per SM, one wave) 33 / 12; K 256, 4096 x 256 (13, one) 57 / 27; K 1024, SwiGLU, 192 x 4096
    // (20, two) 182 / 207, 512 (54, four) 451 / 404; K 2048, 512 x 3072 (20, two) 370 / 288.
    const int tok = g.a2 ? 32 : 64, limit = g.a2 && g.k <= 64 ? 4 : g.k <= 192 ? 6 : g.a2 ? 11 : 10;
    const long long sms = c->num_sms, tiles = (long long)n_tiles * g.groups * ((g.m_tok + tok - 1) / tok);
    if (warp_ctas > limit * ((tiles + sms - 1) / sms) * sms) {
        if (g.k <= 128) return tiled(g.a2 ? gemm_simt_tiled_kernel<T, true, 32, true> : gemm_simt_tiled_kernel<T, false, 64, true>, tok);
        return tiled(g.a2 ? gemm_simt_tiled_kernel<T, true, 32, false> : gemm_simt_tiled_kernel<T, false, 64, false>, tok);
    }
    // Few token rows under many weight rows at a short K: tiles of 16 tokens, from three CTAs per SM of the warp-per-rows
    // form at K 64 and twelve at 128 and 192 (above 8 tokens there), and where 128 rows are mostly not padding.
    // Measured, warp-per-rows / these: K 64, 30 rows x 8192 (3.4 CTAs per SM) 12.2 / 10.1, 15 x 32000 (6.6) 18.4 / 12.2; K 128,
    // 7 x 32000 (6.6) 16.4 / 18.4, 7 x 151936 (31) 59 / 55; K 192, 7 x 151936 65 / 80, 15 rows 105 / 82.
    const long long tiles16 = (long long)n_tiles * g.groups * ((g.m_tok + 15) / 16);
    if (!g.a2 && g.k <= 192 && (g.k <= 128 || g.m_tok > 8) && warp_ctas > 3 * std::max(tiles16, (g.k <= 64 ? 1 : 4) * sms))
        return tiled(gemm_simt_tiled_kernel<T, false, 16, true>, 16);
    return launch_kernel(c->pdl, tt == 8 ? gemm_simt_kernel<T, 8> : gemm_simt_kernel<T, 16>,
                         dim3(n_slices * g.groups, (g.m_tok + tt - 1) / tt), dim3(kSimtThreads), 0, s,
                         (const T*)g.a, (const T*)g.a2, (const T*)g.b, g.n, g.k, g.m_tok, a_gr, g.b_group_rows,
                         g.b_shared, g.b_kgroup, n_slices, g.ep);
}

}  // namespace

cudaError_t launch_gemm_simt(dflare_ctx* c, const GemmDesc& g, cudaStream_t s) {
    if (g.m_tok <= 0 || g.n <= 0) return cudaSuccess;
    if (g.b_kgroup > 0 && (g.k % g.b_kgroup != 0 || g.groups != 1)) return cudaErrorInvalidValue;
    return c->cfg.dtype == DFLARE_F32 ? launch_t<float>(c, g, s) : launch_t<bf16>(c, g, s);
}

}  // namespace dfl
