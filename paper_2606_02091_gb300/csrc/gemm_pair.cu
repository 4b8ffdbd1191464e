// Projection GEMM for many token rows on pairs of SMs (tcgen05 cta_group::2 + TMEM + TMA).
//
// From about 128 token rows on, a projection is no longer bound by the weights' HBM time alone: with
// one CTA per 128-feature tile every k-block of 64 brings 16 KB of weights and up to 32 KB of tokens
// into shared memory and is read from there once per MMA, which is more than shared memory and the
// L2-to-SM path carry at the tensor cores' rate. Here two CTAs of a cluster share one tile of 256
// token rows x bn features (M 256): each keeps 128 token rows and half of the features, and the
// pair's tensor cores read both halves of the features, so a 256 x 256 tile needs 32 KB per k-block
// and SM instead of 48. The tokens are the M operand here (the swapped order of the decode GEMM
// exists for token tiles smaller than 128): the tile's features can be any multiple of 64, so that
// one wave of pairs covers the chip, and a thread of the epilogue holds one token's features.
//
// Measured (bf16, back to back, against the single-SM GEMM): 2560 rows x 16384 x 4096 263 -> 215 us
// (1597 TFLOP/s, 0.83 of cuBLAS's burst rate); gate/up of one layer at 256 rows 55 -> 38 us (203 MB of
// weights: 5.3 TB/s). Bound by the tensor cores in a context fill, by HBM and the fixed parts of a launch at 256
// rows.
//
// Work unit = (group, feature tile, 256-token tile, K split), walked by a persistent grid of pairs. Per
// CTA (320 threads):
//   warps 0-7  epilogue: tcgen05.ld (warp w: token rows 32 (w % 4) .. of this CTA's 128, every second
//              32- or 64-feature chunk), staged per warp in a swizzled 4 KB box and written by one
//              TMA store, or added in L2 by one TMA reduction (residual and Q/K^d/V^d sums: full
//              lines instead of 16-byte reductions per thread); context keys and values go from the
//              registers to their cache rows.
//   warp 8     TMA producer of this CTA's token and feature rows; both CTAs' copies complete on the
//              even CTA's barrier. The first ring's weights are requested before the dependency wait.
//   warp 9     TMEM allocation; in the even CTA one thread issues the pair's MMAs and commits the
//              stages and accumulators to both CTAs.
// Every wait on an mbarrier is bounded (2 s); on a timeout the CTA sets DFLARE_DEVERR_TIMEOUT, stops
// issuing work, drains, meets its peer at the cluster barrier and frees its TMEM.
#include <algorithm>
#include <cstring>

#include "epilogue.cuh"
#include "internal.h"
#include "umma.cuh"

namespace dfl {
namespace {

constexpr int kPairThreads = 320;
constexpr int kPairTok = 256;                 // token rows of a unit, 128 per CTA
constexpr int kPairBK = 64;
constexpr int kPairMaxStages = 8;
constexpr int kPairEpiWarps = 8;
constexpr int kPairMaxTokList = 4096;         // token tiles a compacted launch can list (2^20 rows)
constexpr uint32_t kTokBytes = 128 * kPairBK * 2;
constexpr uint32_t kBoxBytes = 4096;          // a warp's staging box: 32 rows x 128 bytes
constexpr int kPairSmemLimit = 227 * 1024;

struct PairArgs {
    CUtensorMap map_t, map_w, map_w2, map_o;   // tokens, weights, up weights (SwiGLU), output
    int n_units, n_tiles, tok_tiles, splits, kb_per_split, k_blocks;
    int bn, n_a, stages, n_bufs, kbs, compact, evict_first;
    uint32_t w_bytes, stage_bytes, idesc;      // w_bytes: one CTA's half of a feature tile's k-block
    int t_kg;                  // > 0: token group z holds k-blocks [z t_kg, (z+1) t_kg)
    int t_gsel;                // 1: token group = weight group; 0: one token group for all
    uint32_t* err;
    EpiParams ep;
    unsigned long long* t_stamps;
    int t_slots;
};

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t map_rank0(uint32_t saddr) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(saddr));
    return r;
}
__device__ __forceinline__ void arrive_cluster(uint32_t bar) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// a copy into this CTA's shared memory that completes on a barrier of the pair's even CTA
__device__ __forceinline__ void tma_load_pair(uint32_t dst, const CUtensorMap* map, int row, int kb, int z,
                                              uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(row), "r"(kb), "r"(z), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void tma_load_pair_hint(uint32_t dst, const CUtensorMap* map, int row, int kb, int z,
                                                   uint32_t bar, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        ".L2::cache_hint [%0], [%1, {%2, %3, %4, %5}], [%6], %7;" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(row), "r"(kb), "r"(z), "r"(bar), "l"(policy)
        : "memory");
}
__device__ __forceinline__ void umma_pair(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}
// arrives on the barrier at this offset in both CTAs of the pair
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
        "h"((uint16_t)3)
        : "memory");
}

struct PairUnit {
    int group, n_tile, tok_tile, kb0, kb1;
};

__global__ void __launch_bounds__(kPairThreads, 1) gemm_pair_kernel(const __grid_constant__ PairArgs args) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t pad = (1024u - (raw & 1023u)) & 1023u;
    uint8_t* smem = smem_raw + pad;
    const uint32_t sbase = raw + pad;
    const int S = args.stages, kbs = args.kbs, bn = args.bn, n_a = args.n_a, n_bufs = args.n_bufs;
    const uint32_t stage_bytes = args.stage_bytes, w_bytes = args.w_bytes;
    uint32_t* const err = args.err;
    const uint32_t box0 = sbase + (uint32_t)S * stage_bytes;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + (size_t)S * stage_bytes + kPairEpiWarps * kBoxBytes);
    uint32_t* misc = reinterpret_cast<uint32_t*>(bars + 2 * S + 5);
    const uint32_t bar0 = smem_u32(bars);
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (S + s); };
    auto tfull_bar = [&](int b) { return bar0 + 8u * (2 * S + b); };
    auto tempty_bar = [&](int b) { return bar0 + 8u * (2 * S + 2 + b); };
    const uint32_t drain_bar = bar0 + 8u * (2 * S + 4);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)cluster_rank();
    const int pair0 = (int)(blockIdx.x >> 1), n_pairs = (int)(gridDim.x >> 1);
    unsigned long long* const tst = args.t_stamps;
    if (tst && threadIdx.x == 0) atomicMin(tst, (unsigned long long)globaltimer_ns());
    if (warp == 8 && lane == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&args.map_t)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&args.map_w)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&args.map_w2)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&args.map_o)) : "memory");
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(full_bar(s), 1);
            mbar_init(empty_bar(s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(tfull_bar(b), 1);
            mbar_init(tempty_bar(b), 2 * kPairEpiWarps);
        }
        mbar_init(drain_bar, 1);
        misc[1] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    // a context fill of sequences with different lengths: units run over the token tiles that hold appended
    // rows, listed in shared memory (both CTAs of a pair form the same list), not over the padding
    int* const tok_list = reinterpret_cast<int*>(misc + 4);
    if (args.compact) {
        pdl_wait();
        if (tst && threadIdx.x == 0) atomicMin(tst + args.t_slots, (unsigned long long)globaltimer_ns());
        if (warp == 0) {
            const int nm = args.ep.n_max;
            int cnt = 0;
            for (int base = 0; base < args.tok_tiles; base += 32) {
                const int tt = base + lane;
                bool v = false;
                if (tt < args.tok_tiles) {
                    const int r0 = tt * kPairTok, r1 = min(args.ep.m_tok, r0 + kPairTok);
                    for (int b = r0 / nm; b <= (r1 - 1) / nm && !v; ++b)
                        v = args.ep.app_cnt[b] > max(0, r0 - b * nm);
                }
                const unsigned m = __ballot_sync(0xffffffffu, v);
                if (v) tok_list[cnt + __popc(m & ((1u << lane) - 1u))] = tt;
                cnt += __popc(m);
            }
            if (lane == 0) misc[3] = (uint32_t)cnt;
        }
    }
    if (warp == 9) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&misc[0]))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_barrier();   // both CTAs' barriers are initialised
    tc_fence_after();
    const uint32_t tmem = misc[0];
    volatile int* abort_flag = reinterpret_cast<volatile int*>(&misc[1]);
    int n_units = args.n_units, tok_tiles = args.tok_tiles;
    if (args.compact) {
        n_units = n_units / tok_tiles * (int)misc[3];
        tok_tiles = (int)misc[3];
    }
    auto unit = [&](int u) {
        PairUnit x;
        const int split = u % args.splits;
        int t = u / args.splits;
        x.tok_tile = t % tok_tiles;
        if (args.compact) x.tok_tile = tok_list[x.tok_tile];
        t /= tok_tiles;
        x.n_tile = t % args.n_tiles;
        x.group = t / args.n_tiles;
        x.kb0 = split * args.kb_per_split;
        x.kb1 = min(args.k_blocks, x.kb0 + args.kb_per_split);
        return x;
    };
    const int acc_cols = n_a * bn;
    const uint32_t w_base = kTokBytes * (uint32_t)kbs;   // the stage: the token rows' kbs k-blocks, then the weights'

    if (warp == 8) {
        if (elect_one()) {
            // ---------------- TMA producer
            uint64_t policy = 0;
            const bool evict_first = args.evict_first != 0;
            if (evict_first) asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
            int stage = 0, npend = 0;
            uint32_t phase = 0, issued = 0, issued_phase = 0;
            bool ok = true, waited = args.compact != 0;
            const uint32_t tx = 2u * stage_bytes;   // both CTAs
            int pend_kb[kPairMaxStages], pend_tok[kPairMaxStages], pend_grp[kPairMaxStages];
            auto load_w = [&](uint32_t dst, const CUtensorMap* map, int row, int kb, int z, uint32_t bar) {
                if (evict_first)
                    tma_load_pair_hint(dst, map, row, kb, z, bar, policy);
                else
                    tma_load_pair(dst, map, row, kb, z, bar);
            };
            auto load_t = [&](int st, int kb, int tok_tile, int group) {
                int z = group * args.t_gsel;
                if (args.t_kg > 0) {
                    z = kb / args.t_kg;
                    kb -= z * args.t_kg;
                }
                tma_load_pair(sbase + (uint32_t)st * stage_bytes, &args.map_t, tok_tile * kPairTok + rank * 128, kb, z,
                              map_rank0(full_bar(st)));
            };
            auto flush = [&] {
                pdl_wait();
                if (tst) atomicMin(tst + args.t_slots, (unsigned long long)globaltimer_ns());
                waited = true;
                for (int i = 0; i < npend; ++i) load_t(i, pend_kb[i], pend_tok[i], pend_grp[i]);
            };
            for (int u = pair0; u < n_units && ok; u += n_pairs) {
                const PairUnit x = unit(u);
                const int row = x.n_tile * bn + rank * (bn >> 1);
                for (int kb = x.kb0; kb < x.kb1; kb += kbs) {
                    if (!bar_wait(empty_bar(stage), phase ^ 1u, abort_flag, err)) {
                        ok = false;
                        break;
                    }
                    const uint32_t st = sbase + (uint32_t)stage * stage_bytes + w_base;
                    const uint32_t bar = map_rank0(full_bar(stage));
                    if (rank == 0) mbar_expect_tx(full_bar(stage), tx);
                    load_w(st, &args.map_w, row, kb, x.group, bar);
                    if (n_a == 2) load_w(st + (uint32_t)kbs * w_bytes, &args.map_w2, row, kb, x.group, bar);
                    if (waited) {
                        load_t(stage, kb, x.tok_tile, x.group);
                    } else {   // the first ring: slots 0, 1, ... in order
                        pend_kb[npend] = kb;
                        pend_tok[npend] = x.tok_tile;
                        pend_grp[npend] = x.group;
                        if (++npend == S) flush();
                    }
                    issued |= 1u << stage;
                    issued_phase = (issued_phase & ~(1u << stage)) | (phase << stage);
                    if (++stage == S) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
            }
            if (!waited) flush();
            // No copy is still landing and no commit still arriving in this CTA's shared memory when it leaves: a
            // stage's empty barrier completes after the MMAs that read both CTAs' copies of it (the odd CTA's
            // copies complete on the even one's barrier), and the last commit arrives in both CTAs, of which the
            // even one's issuing thread sees its own. The cluster barrier below orders what the threads of the
            // pair did, not these arrivals. After a timeout some stages have no MMAs any more; one limit for all
            // of them ends the wait.
            volatile int never = 0;
            for (int s = 0; s < S; ++s)
                if (issued & (1u << s)) bar_wait_slow(empty_bar(s), (issued_phase >> s) & 1u, &never, err);
            if (rank == 1) bar_wait_slow(drain_bar, 0, &never, err);
        }
    } else if (warp == 9) {
        if (rank == 0 && elect_one()) {
            // ---------------- MMA issuer of the pair
            int stage = 0, acc = 0;
            uint32_t phase = 0, acc_phase = 0;
            bool ok = true;
            for (int u = pair0; u < n_units && ok; u += n_pairs) {
                const PairUnit x = unit(u);
                if (!bar_wait(tempty_bar(acc), acc_phase ^ 1u, abort_flag, err)) break;
                tc_fence_after();
                const uint32_t d0 = tmem + (uint32_t)(acc * acc_cols);
                for (int kb = x.kb0; kb < x.kb1; kb += kbs) {
                    const int nk = min(kbs, x.kb1 - kb);
                    if (!bar_wait(full_bar(stage), phase, abort_flag, err)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t st = sbase + (uint32_t)stage * stage_bytes;
                    for (int j = 0; j < nk; ++j) {
                        const uint64_t dt = smem_desc(st + j * kTokBytes);
                        const uint64_t dw = smem_desc(st + w_base + (uint32_t)j * w_bytes);
                        const uint64_t dw2 = smem_desc(st + w_base + (uint32_t)(kbs + j) * w_bytes);
#pragma unroll
                        for (int k = 0; k < kPairBK / 16; ++k) {
                            const uint32_t accum = (kb > x.kb0 || j > 0 || k > 0) ? 1u : 0u;
                            umma_pair(d0, dt + 2 * k, dw + 2 * k, args.idesc, accum);
                            if (n_a == 2) umma_pair(d0 + bn, dt + 2 * k, dw2 + 2 * k, args.idesc, accum);
                        }
                    }
                    umma_commit_pair(empty_bar(stage));
                    if (++stage == S) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
                if (!ok) break;
                umma_commit_pair(tfull_bar(acc));
                if (n_bufs == 2) {
                    acc ^= 1;
                    if (acc == 0) acc_phase ^= 1u;
                } else {
                    acc_phase ^= 1u;
                }
            }
            // all issued MMAs complete before either CTA's TMEM is released
            umma_commit_pair(drain_bar);
            volatile int never = 0;
            bar_wait(drain_bar, 0, &never, err);
        }
    } else {
        // ---------------- epilogue warps: lane = token row
        pdl_wait();
        // dependents may start once every CTA has passed its own dependency wait (see the single-SM GEMM)
        if (threadIdx.x == 0) pdl_trigger();
        const EpiParams& ep = args.ep;
        const int quarter = warp & 3, half = warp >> 2;
        const uint32_t box = box0 + (uint32_t)warp * kBoxBytes;
        uint8_t* const box_row = smem + (box - sbase) + lane * 128;
        const bool red = ep.kind == EPI_RESID || ep.kind == EPI_RED32;
        bool in_flight = false;   // lane 0's last store may still be reading the box
        auto box_free = [&] {
            if (in_flight && lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            in_flight = true;
            __syncwarp();
        };
        auto box_out = [&](int n0, int tok0, int group) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) {
                if (red)
                    tma_reduce(&args.map_o, box, n0, tok0, group);
                else
                    tma_store(&args.map_o, box, n0, tok0, group);
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
        };
        // 32 values as bf16 into 16-byte chunks [4 hc, 4 hc + 4) of this lane's 128-byte box row
        auto box_bf16 = [&](const float* v, int hc) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                store8(reinterpret_cast<bf16*>(box_row + (((4 * hc + j) ^ (lane & 7)) << 4)), v + 8 * j);
        };
        int acc = 0;
        uint32_t acc_phase = 0;
        for (int u = pair0; u < n_units; u += n_pairs) {
            const PairUnit x = unit(u);
            const bool got = bar_wait(tfull_bar(acc), acc_phase, abort_flag, err);
            if (!__all_sync(0xffffffffu, got)) break;
            tc_fence_after();
            const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * acc_cols);
            const int tok0 = x.tok_tile * kPairTok + rank * 128 + quarter * 32;   // this warp's 32 token rows
            const int nb = x.n_tile * bn;
            if (tok0 < ep.m_tok) {
                if (red || ep.kind == EPI_F32) {
                    for (int c = half; c < bn / 32; c += 2) {
                        if (nb + c * 32 >= ep.n) break;
                        float v[32];
                        tmem_ld32(taddr + (uint32_t)(c * 32), v);
                        box_free();
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            *reinterpret_cast<float4*>(box_row + ((j ^ (lane & 7)) << 4)) =
                                make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
                        box_out(nb + c * 32, tok0, 0);
                    }
                } else if (ep.kind == EPI_SWIGLU) {
                    for (int c = half; c < bn / 64; c += 2) {
                        if (nb + c * 64 >= ep.n) break;
                        box_free();
#pragma unroll
                        for (int hc = 0; hc < 2; ++hc) {
                            float v[32], up[32];
                            tmem_ld32(taddr + (uint32_t)(c * 64 + hc * 32), v);
                            tmem_ld32(taddr + (uint32_t)(bn + c * 64 + hc * 32), up);
#pragma unroll
                            for (int i = 0; i < 32; ++i) v[i] = silu_f(v[i]) * up[i];
                            box_bf16(v, hc);
                        }
                        box_out(nb + c * 64, tok0, 0);
                    }
                } else if (ep.kind == EPI_STORE) {
                    for (int c = half; c < bn / 64; c += 2) {
                        if (nb + c * 64 >= ep.n) break;
                        box_free();
#pragma unroll
                        for (int hc = 0; hc < 2; ++hc) {
                            float v[32];
                            tmem_ld32(taddr + (uint32_t)(c * 64 + hc * 32), v);
                            if (ep.bias) {
                                const bf16* bias = reinterpret_cast<const bf16*>(ep.bias) +
                                                   (size_t)x.group * ep.n + nb + c * 64 + hc * 32;
#pragma unroll
                                for (int j = 0; j < 4; ++j) {
                                    float bv[8];
                                    load8(bias + 8 * j, bv);
#pragma unroll
                                    for (int e = 0; e < 8; ++e) v[8 * j + e] += bv[e];
                                }
                            }
                            box_bf16(v, hc);
                        }
                        box_out(nb + c * 64, tok0, x.group);
                    }
                } else if (ep.kind == EPI_KV_APPEND) {
                    const int hd = ep.head_dim, hh = hd >> 1;
                    const int tok = tok0 + lane;
                    const int b = min(tok, ep.m_tok - 1) / ep.n_max, r = tok - b * ep.n_max;
                    const bool live = tok < ep.m_tok && r < ep.app_cnt[b];
                    const int pos = live ? ep.app_base[b] + r : 0;
                    const int hkv = ep.d_kv / hd;
                    // item = 32 head dims and their rotary partners, hd / 2 further (a head's 64 or
                    // 128 features lie in one unit: bn is a multiple of 128, d_kv of 128)
                    if (__any_sync(0xffffffffu, live))
                        for (int c = half; c < bn / 64; c += 2) {
                            const int per = hd / 64, c_lo = (c / per) * hd + (c % per) * 32;   // unit column
                            const int n0 = nb + c_lo;
                            if (n0 >= ep.n) break;
                            const bool is_k = n0 < ep.d_kv;
                            const int col = is_k ? n0 : n0 - ep.d_kv;
                            const int g = col / hd, j0 = col - g * hd;
                            float v[32], y[32];
                            tmem_ld32(taddr + (uint32_t)c_lo, v);
                            tmem_ld32(taddr + (uint32_t)(c_lo + hh), y);
                            if (live) {
                                if (is_k) {
                                    const float4* cp = reinterpret_cast<const float4*>(ep.rope_cos + (size_t)pos * hh + j0);
                                    const float4* sp = reinterpret_cast<const float4*>(ep.rope_sin + (size_t)pos * hh + j0);
                                    float4 cs[8], sn[8];
#pragma unroll
                                    for (int j = 0; j < 8; ++j) {
                                        cs[j] = __ldg(cp + j);
                                        sn[j] = __ldg(sp + j);
                                    }
                                    const float* cf = reinterpret_cast<const float*>(cs);
                                    const float* sf = reinterpret_cast<const float*>(sn);
#pragma unroll
                                    for (int i = 0; i < 32; ++i) {
                                        const float a = v[i], d2 = y[i];
                                        v[i] = a * cf[i] - d2 * sf[i];
                                        y[i] = d2 * cf[i] + a * sf[i];
                                    }
                                }
                                bf16* dst = reinterpret_cast<bf16*>(is_k ? ep.kcache : ep.vcache) +
                                            ((((size_t)x.group * ep.max_batch + b) * hkv + g) * ep.max_ctx + pos) * hd + j0;
#pragma unroll
                                for (int j = 0; j < 4; ++j) store8(dst + 8 * j, v + 8 * j);
#pragma unroll
                                for (int j = 0; j < 4; ++j) store8(dst + hh + 8 * j, y + 8 * j);
                            }
                            __syncwarp();   // the next item's loads are warp-collective
                        }
                }
            }
            __syncwarp();
            tc_fence_before();
            if (lane == 0) arrive_cluster(map_rank0(tempty_bar(acc)));
            if (n_bufs == 2) {
                acc ^= 1;
                if (acc == 0) acc_phase ^= 1u;
            } else {
                acc_phase ^= 1u;
            }
        }
        // the copies have read the staging boxes before the CTA's shared memory goes (what they write is
        // visible to the dependents with the end of the grid, as any store's)
        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
    }
    __syncwarp();
    __syncthreads();
    if (tst && threadIdx.x == 0) atomicMax(tst + 2 * args.t_slots, (unsigned long long)globaltimer_ns());
    // neither CTA leaves, or frees its tensor memory, while the other's threads or MMAs may touch it
    cluster_barrier();
    if (warp == 9) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    }
}

// Tile width and K splits of a launch by the estimated clocks of its busiest pair. Per 64-wide k-block a
// pair is bound by its MMAs (max(bn / 2, 64) clocks per 16 of K and accumulator) or by the bytes each SM takes
// from L2 (16 KB of tokens and n_a bn / 2 weight rows, about 60 bytes per clock).
struct PairPlan {
    int bn, splits, kb_per_split;
};
PairPlan plan_pair(const GemmDesc& g, int pairs, bool may_split) {
    const int kb = (g.k + kPairBK - 1) / kPairBK, n_a = g.a2 ? 2 : 1;
    const int tt = (g.m_tok + kPairTok - 1) / kPairTok;
    const int step = g.ep.kind == EPI_KV_APPEND ? 128 : 64;
    PairPlan best{step, 1, kb};
    double best_t = 1e30;
    for (int bn = step; bn <= 256; bn += step) {
        const long long tiles = (long long)g.groups * ((g.n + bn - 1) / bn) * tt;
        const double per_kb = std::max(4.0 * n_a * std::max(bn / 2, 64), (16384.0 + n_a * bn * 64.0) / 60.0);
        const bool overlap = 2 * n_a * bn <= 512;
        const double epi = 1500.0 + 12.0 * bn * n_a;
        for (int sp = 1; sp <= (may_split ? 8 : 1) && sp <= kb / 4 + 1; ++sp) {
            const int kbp = (kb + sp - 1) / sp, spn = (kb + kbp - 1) / kbp;
            const long long waves = (tiles * spn + pairs - 1) / pairs;
            const double main = kbp * per_kb;
            const double t = waves * (overlap ? std::max(main, epi) : main + epi) + (overlap ? epi : 0) + 2000.0;
            if (t < best_t) {
                best_t = t;
                best = {bn, spn, kbp};
            }
        }
    }
    return best;
}

}  // namespace

bool gemm_pair_fits(const dflare_ctx* c, const GemmDesc& g) {
    const EpiParams& ep = g.ep;
    // Against the single-SM GEMM at d 4096, ffn 12288 (us, single -> pair): 256 rows Q/K/V 16.8 -> 16.6,
    // O 14.2 -> 14.2, down 27.5 -> 25.9, gate/up 47.8 -> 38.0, LM head (40000 entries) 88.6 -> 68.3; 224 rows
    // 16.1 -> 16.6, 13.5 -> 14.1, 26.2 -> 25.8, 44.8 -> 37.8, 84.7 -> 67.7; 144 rows 13.9 -> 16.5, 11.7 -> 14.1,
    // 22.2 -> 25.6, 37.3 -> 37.6, 64.6 -> 67.1. The projections that split K over all SMs cross over near 224
    // rows, an LM head of several waves at 160 (65.8 -> 67.1, at 192 rows 77.8 -> 67.4), the others at about 128
    // (gate/up of the Qwen3-4B shape, 144 rows: 23.0 -> 21.8; 4096 logits 21.6 -> 16.7).
    const int from = ep.kind == EPI_RESID || ep.kind == EPI_RED32 ? 224
                     : ep.kind == EPI_F32 && g.n >= 128 * c->num_sms ? 160 : 128;
    if (g.m_tok <= from || g.n % 4 != 0 || g.k % kPairBK != 0) return false;
    if ((g.m_tok + kPairTok - 1) / kPairTok > kPairMaxTokList) return false;
    switch (ep.kind) {
        case EPI_F32: return ep.ldo % 4 == 0 && (reinterpret_cast<uintptr_t>(ep.out) & 15u) == 0;
        case EPI_RED32: return ep.ldo % 4 == 0;
        case EPI_RESID: return ep.ld_resid % 4 == 0;
        case EPI_SWIGLU: return g.n % 8 == 0 && ep.ldo % 8 == 0;
        case EPI_STORE:
            return g.n % 64 == 0 && ep.ldo % 8 == 0 && ep.out_gstride % 8 == 0 &&
                   (reinterpret_cast<uintptr_t>(ep.out) & 15u) == 0 && (reinterpret_cast<uintptr_t>(ep.bias) & 15u) == 0;
        case EPI_KV_APPEND: return g.n % 128 == 0;
        default: return false;
    }
}

cudaError_t launch_gemm_pair(dflare_ctx* c, const GemmDesc& g, cudaStream_t s, std::string* why) {
    PairArgs a;
    memset(&a, 0, sizeof(a));
    const bool det = c->cfg.flags & DFLARE_FLAG_DETERMINISTIC;
    const int pairs = c->num_sms / 2;
    const bool may_split = g.ep.kind == EPI_RED32 || (g.ep.kind == EPI_RESID && !det);
    const PairPlan p = plan_pair(g, pairs, may_split);
    a.bn = p.bn;
    a.n_a = g.a2 ? 2 : 1;
    a.splits = p.splits;
    a.kb_per_split = p.kb_per_split;
    a.k_blocks = (g.k + kPairBK - 1) / kPairBK;
    a.n_tiles = (g.n + a.bn - 1) / a.bn;
    a.tok_tiles = (g.m_tok + kPairTok - 1) / kPairTok;
    a.n_units = g.groups * a.n_tiles * a.tok_tiles * a.splits;
    a.compact = (g.ep.kind == EPI_KV_APPEND && a.tok_tiles > 1) ? 1 : 0;
    a.w_bytes = (uint32_t)a.bn / 2 * kPairBK * 2;
    const uint32_t kb_bytes = kTokBytes + (uint32_t)a.n_a * a.w_bytes;
    const int fixed = 1024 + kPairEpiWarps * (int)kBoxBytes + 8 * (2 * kPairMaxStages + 5) + 16 +
                      (a.compact ? 4 * a.tok_tiles : 0);
    const int budget = kPairSmemLimit - fixed;
    a.kbs = budget / (int)(2 * kb_bytes) >= 3 ? 2 : 1;
    if (g.b_kgroup > 0 && g.b_kgroup / kPairBK % a.kbs != 0) a.kbs = 1;   // a copy stays within one token group
    a.stage_bytes = kb_bytes * (uint32_t)a.kbs;
    a.stages = std::min(kPairMaxStages, budget / (int)a.stage_bytes);
    if (a.stages < 2) {
        if (why) *why = "two-SM GEMM: tile does not fit in shared memory";
        return cudaErrorInvalidValue;
    }
    a.n_bufs = 2 * a.n_a * a.bn <= 512 ? 2 : 1;
    // tokens that pass once leave their weights no second reader
    a.evict_first = a.tok_tiles == 1;
    // kind::f16 instruction descriptor: fp32 accumulate, bf16 A and B, both K-major, N = bn, M = 256
    a.idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(a.bn >> 3) << 17) | ((256u >> 4) << 24);
    a.t_kg = g.b_kgroup / kPairBK;
    a.t_gsel = g.b_shared ? 0 : 1;
    a.err = c->err;
    a.ep = g.ep;
    const uint64_t k = (uint64_t)g.k, b_k = g.b_kgroup > 0 ? (uint64_t)g.b_kgroup : k;
    const uint64_t b_groups = g.b_kgroup > 0 ? k / b_k : (g.b_shared ? 1 : g.groups);
    const uint64_t b_rows = (uint64_t)(g.b_group_rows > 0 ? g.b_group_rows : g.m_tok);
    const uint64_t a_rows = (uint64_t)(g.a_group_rows > 0 ? g.a_group_rows : g.n);
    if (g.b_kgroup > 0 && (g.b_kgroup % kPairBK != 0 || g.k % g.b_kgroup != 0 || g.groups != 1)) {
        if (why) *why = "two-SM GEMM: b_kgroup must be a multiple of 64 that divides k, with one group";
        return cudaErrorInvalidValue;
    }
    // [rows][k] operands seen as [k / 64][rows][64], so that one copy brings a stage's kbs k-blocks of an
    // operand in the order in which the MMAs read them (k-blocks past the end read as zeros)
    const uint32_t kbs = (uint32_t)a.kbs;
    const uint32_t t_box[4] = {kPairBK, 128, kbs, 1}, w_box[4] = {kPairBK, (uint32_t)a.bn / 2, kbs, 1};
    const uint64_t t_dims[4] = {kPairBK, (uint64_t)g.m_tok, b_k / kPairBK, b_groups};
    const uint64_t w_dims[4] = {kPairBK, (uint64_t)g.n, k / kPairBK, (uint64_t)g.groups};
    const uint64_t t_st[3] = {b_k * 2, kPairBK * 2, b_rows * b_k * 2}, w_st[3] = {k * 2, kPairBK * 2, a_rows * k * 2};
    bool ok = encode_tma_bf16(&a.map_t, g.b, 4, t_dims, t_st, t_box) &&
              encode_tma_bf16(&a.map_w, g.a, 4, w_dims, w_st, w_box) &&
              encode_tma_bf16(&a.map_w2, g.a2 ? g.a2 : g.a, 4, w_dims, w_st, w_box);
    // the output: boxes of 32 token rows x 128 bytes (context keys and values need no map)
    uint64_t o_dims[3] = {(uint64_t)g.n, (uint64_t)g.m_tok, 1};
    if (g.ep.kind == EPI_RESID || g.ep.kind == EPI_RED32 || g.ep.kind == EPI_F32) {
        const uint64_t ld = (uint64_t)(g.ep.kind == EPI_RESID ? g.ep.ld_resid : g.ep.ldo) * 4;
        const uint64_t st[2] = {ld, ld * (uint64_t)g.m_tok};
        const uint32_t box[3] = {32, 32, 1};
        ok = ok && encode_tma_f32(&a.map_o, g.ep.kind == EPI_RESID ? static_cast<void*>(g.ep.resid) : g.ep.out, 3, o_dims, st, box);
    } else if (g.ep.kind == EPI_SWIGLU || g.ep.kind == EPI_STORE) {
        const uint64_t ld = (uint64_t)g.ep.ldo * 2;
        const bool grouped = g.ep.out_gstride > 0;
        if (grouped) o_dims[2] = (uint64_t)g.groups;
        const uint64_t st[2] = {ld, grouped ? (uint64_t)g.ep.out_gstride * 2 : ld * (uint64_t)g.m_tok};
        const uint32_t box[3] = {64, 32, 1};
        ok = ok && encode_tma_bf16(&a.map_o, g.ep.out, 3, o_dims, st, box);
    } else {
        a.map_o = a.map_t;
    }
    if (!ok) {
        if (why) *why = "cuTensorMapEncodeTiled failed (alignment or driver entry point)";
        return cudaErrorInvalidValue;
    }
    static PerDeviceOnce configured;
    const cudaError_t ce = configured([] {
        return cudaFuncSetAttribute(gemm_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kPairSmemLimit);
    });
    if (ce != cudaSuccess) return ce;
    if (c->t_stamps && c->t_next < c->t_slots) {
        a.t_stamps = c->t_stamps + c->t_next++;
        a.t_slots = c->t_slots;
    }
    const int smem = fixed + a.stages * (int)a.stage_bytes;
    return launch_cluster(c->pdl, 2, gemm_pair_kernel, dim3(2 * std::min(a.n_units, pairs)), dim3(kPairThreads),
                          (size_t)smem, s, a);
}

}  // namespace dfl
