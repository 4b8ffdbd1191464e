// Weight-streaming projection GEMM on the sm_103a tensor cores (tcgen05 + TMEM + TMA).
//
// Every projection of the draft path (context K/V of Eq. 4, Q/K^d/V^d, attention output, SwiGLU
// gate/up and down, LM head) multiplies a few activation rows (batch * B tokens, at most a few
// hundred) by a large weight matrix, so each weight byte is used only m_tok times: the kernel is
// bound by HBM bandwidth while m_tok is below ~280. The layout is therefore "swap AB": the
// 128-row UMMA M dimension runs over weight rows (output features) and the small token count is
// the UMMA N dimension (16..256), so one instruction covers a 128 x bn x 16 piece.
//
// Work unit = (group, 128-feature tile, token tile, K split); for a large LM head over 113 or more token
// rows, a pair of adjacent 128-feature tiles (two accumulators over one activation tile). A
// persistent grid of one CTA per SM walks the units. Per CTA (192 threads):
//   warp 4    TMA producer: per stage, kbs consecutive 128x64 bf16 weight tiles (+ the up tiles
//             for SwiGLU) and the matching bn x 64 activation tiles, 128-byte swizzled; weights
//             carry an L2 evict-first hint (each byte is read once per step). Weights do not
//             depend on the previous kernel: the first ring of stages gets its weight tiles
//             before griddepcontrol.wait, the activation tiles after it.
//   warp 5    allocates TMEM, issues tcgen05.mma (one thread), commits stages back to the
//             producer and finished accumulators to the epilogue; two accumulator buffers let
//             the next unit's MMAs overlap the current unit's epilogue.
//   warps 0-3 epilogue: tcgen05.ld of the accumulator (thread t = TMEM lane t = feature t),
//             split-K reduction through a global workspace (the last CTA of a tile sums the
//             partials in split order, so results are deterministic) where the splits do not add
//             into fp32 sums, then the result: through each warp's own staging slots and TMA (sums,
//             SwiGLU, logits), else turned token-major by the four warps together (apply_epilogue).
//             Measured for the staged form against the other: one launch at 64 tokens, d 4096,
//             gate/up 38.0 -> 34.4 us, O 9.6 -> 8.9, down 20.0 -> 18.5; Qwen3-8B block b4 1008 -> 971.
// Every wait on an mbarrier is bounded (2 s); on a timeout the CTA sets DFLARE_DEVERR_TIMEOUT,
// stops issuing work, drains what it issued and frees its TMEM.
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstring>
#include <mutex>

#include "epilogue.cuh"
#include "umma.cuh"

namespace dfl {
namespace {

constexpr int kThreads = 192;
constexpr int kBM = 128;
constexpr int kBK = 64;
constexpr int kChunk = 16;
constexpr int kMaxStages = 8;
constexpr int kSmemLimit = 227 * 1024;

// How a tile leaves the accumulators. OUT_REGS: chunks of 16 tokens turned token-major in shared memory
// and finished by apply_epilogue. The others: every epilogue warp stages its 32 features of 16 or 32
// tokens in its own slots, token-major, and one TMA copy writes them or adds them in L2: no CTA barrier, no
// per-thread global accesses.
enum OutMode : int {
    OUT_REGS = 0,
    OUT_ADD = 1,      // fp32 sums added to the output (every K split adds its own part, in no fixed order)
    OUT_SWIGLU = 2,   // silu(gate) * up in bf16
    OUT_F32 = 3       // fp32 stored (logits)
};

struct TcArgs {
    CUtensorMap map_a, map_a2, map_b;   // weights, up weights (SwiGLU), activations
    CUtensorMap map_o;                  // output (out_mode != OUT_REGS)
    int n_units, n_tiles, tok_tiles, splits, kb_per_split, k_blocks;
    int bn, n_a, stages, n_bufs, tmem_cols;
    int bm;                    // weight rows of a tile (128; fewer for SwiGLU: see launch_gemm_tc)
    uint32_t a_bytes;          // bytes of one weight sub-tile (bm x 64 bf16)
    int pair;                  // 1: a unit is two adjacent 128-row tiles of one weight matrix
                               // (the second accumulator takes rows 128..255 of the pair)
    int kbs;                   // 64-wide k-blocks per pipeline stage
    uint32_t b_bytes;          // bytes of one activation sub-tile (bn x 64 bf16)
    uint32_t idesc;
    uint32_t stage_bytes;
    float* ws;
    uint32_t* tile_cnt;
    uint32_t* err;
    EpiParams ep;
    // activation addressing of the kAux instance only
    int b_kg;                  // > 0: activation group z holds contraction indices [z b_kg, (z+1) b_kg)
    int b_gsel;                // 1: activation group = weight group; 0: one activation group for all
    int out_mode;              // OutMode: results that leave through staged TMA copies (map_o)
    int n_slots;               // staging slots per epilogue warp
    int epi_bytes;             // staging area (OUT_REGS: [accumulator][16 tokens][128 features] fp32)
    unsigned long long* t_stamps;   // launch timing: entry, dependency met, exit (nullptr: off)
    int t_slots;
};

__device__ __forceinline__ void epi_bar() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

__device__ __forceinline__ uint32_t atom_add_acq_rel(uint32_t* p, uint32_t v) {
    uint32_t old;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}

// The kernel's loop constants, copied out of the parameter block into registers (the block is
// addressed for the tensor maps, so every asm with a memory clobber would otherwise reload them).
struct Geom {
    int n_units, n_tiles, tok_tiles, splits, kb_per_split, k_blocks, n_a, kbs, bn, n_bufs, pair;
    uint32_t a_bytes, b_bytes, stage_bytes, idesc;
};
struct Unit {
    int group, n_tile, tok_tile, split, tile_id, kb0, kb1;
};
__device__ __forceinline__ Unit decode_unit(const Geom& a, int u) {
    Unit x;
    x.split = u % a.splits;
    x.tile_id = u / a.splits;
    int t = x.tile_id;
    x.tok_tile = t % a.tok_tiles;
    t /= a.tok_tiles;
    x.n_tile = t % a.n_tiles;
    x.group = t / a.n_tiles;
    x.kb0 = x.split * a.kb_per_split;
    x.kb1 = min(a.k_blocks, x.kb0 + a.kb_per_split);
    return x;
}

// EPI_RESID with the residual values already in registers: resid[tok][n] += acc.
__device__ __forceinline__ void load_resid(const EpiParams& ep, int n_tile, int tok0, int t, float* r) {
    const int n = n_tile * 128 + t;
    const int nvalid = min(kChunk, ep.m_tok - tok0);
#pragma unroll
    for (int c = 0; c < kChunk; ++c)
        r[c] = (n < ep.n && c < nvalid) ? ep.resid[(size_t)(tok0 + c) * ep.ld_resid + n] : 0.f;
}
__device__ __forceinline__ void resid_epilogue(const EpiParams& ep, const float* tile, int n_tile,
                                               int tok0, int t, const float* r) {
    const int n = n_tile * 128 + t;
    if (n >= ep.n) return;
    const int nvalid = min(kChunk, ep.m_tok - tok0);
#pragma unroll
    for (int c = 0; c < kChunk; ++c)
        if (c < nvalid) ep.resid[(size_t)(tok0 + c) * ep.ld_resid + n] = r[c] + tile[c * 128 + t];
}

// K splits through the workspace: this CTA's partial accumulators of a tile go out ([accumulator][16-token
// chunk][feature][16] per (tile, split)) and the accumulator buffer is released; true for the last CTA of
// the tile to get here, which then finishes it.
__device__ __forceinline__ bool split_partials(const TcArgs& args, const Geom& G, const Unit& x, uint32_t taddr,
                                               uint32_t tempty, uint32_t* misc, int t) {
    const int bn = G.bn, na = G.n_a;
    float* dst = args.ws + (size_t)(x.tile_id * G.splits + x.split) * na * bn * 128;
    for (int a = 0; a < na; ++a)
        for (int c0 = 0; c0 < bn; c0 += kChunk) {
            float v[kChunk];
            tmem_ld16(taddr + (uint32_t)(a * bn + c0), v);
            float4* d4 = reinterpret_cast<float4*>(dst + ((size_t)(a * (bn / kChunk) + c0 / kChunk) * 128 + t) * kChunk);
#pragma unroll
            for (int k = 0; k < kChunk / 4; ++k)
                d4[k] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
        }
    tc_fence_before();
    mbar_arrive(tempty);
    // the CTA barrier orders every thread's partial before thread 0's release; its acquire (when
    // last) orders the other partials before the reads that follow
    epi_bar();
    if (t == 0) {
        const uint32_t prev = atom_add_acq_rel(&args.tile_cnt[x.tile_id], 1u);
        misc[2] = (prev == (uint32_t)(G.splits - 1)) ? 1u : 0u;
        if (prev == (uint32_t)(G.splits - 1)) args.tile_cnt[x.tile_id] = 0;
    }
    epi_bar();
    return misc[2] != 0;
}
// One feature's 16 tokens c0 .. of accumulator a, summed over the splits in split order (deterministic);
// four 16-byte loads per split, several splits in flight.
__device__ __forceinline__ void sum_partials(const float* part, const Geom& G, int na, int a, int c0, int t, float* v) {
    float4 acc4[kChunk / 4];
#pragma unroll
    for (int k = 0; k < kChunk / 4; ++k) acc4[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    const size_t off = ((size_t)(a * (G.bn / kChunk) + c0 / kChunk) * 128 + t) * kChunk;
#pragma unroll 4
    for (int s = 0; s < G.splits; ++s) {
        const float4* src = reinterpret_cast<const float4*>(part + (size_t)s * na * G.bn * 128 + off);
#pragma unroll
        for (int k = 0; k < kChunk / 4; ++k) {
            const float4 w4 = __ldcg(src + k);
            acc4[k].x += w4.x;
            acc4[k].y += w4.y;
            acc4[k].z += w4.z;
            acc4[k].w += w4.w;
        }
    }
#pragma unroll
    for (int k = 0; k < kChunk / 4; ++k) {
        v[4 * k] = acc4[k].x;
        v[4 * k + 1] = acc4[k].y;
        v[4 * k + 2] = acc4[k].z;
        v[4 * k + 3] = acc4[k].w;
    }
}
// A tile's results through this warp's staging slots and TMA (out_mode != OUT_REGS), CH tokens at a time:
// lane = feature 32 warp + lane of the tile, so a token's 32 features are one conflict-free row of a slot
// (128 bytes of fp32 in the copies' 128-byte swizzle, or two boxes of 32 bytes of bf16).
template <int CH>
__device__ __forceinline__ void staged_out(const TcArgs& args, const Geom& G, const Unit& x, uint32_t taddr,
                                           const float* part, float* stage, int warp, int lane) {
    const int bn = G.bn, mode = args.out_mode, t = warp * 32 + lane;
    const bool h16 = mode == OUT_SWIGLU;
    const uint32_t slot_bytes = CH * (h16 ? 64u : 128u);
    uint8_t* const base = reinterpret_cast<uint8_t*>(stage) + (uint32_t)(warp * args.n_slots) * slot_bytes;
    const int n0 = x.n_tile * args.bm + warp * 32, nw = min(32, args.bm - warp * 32);   // features of this warp
    if (nw <= 0) return;
    int slot = 0;
    for (int c0 = 0; c0 < bn; c0 += CH) {
        uint32_t v[CH], up[CH];
        if (part) {
#pragma unroll
            for (int h = 0; h < CH; h += kChunk) {
                sum_partials(part, G, G.n_a, 0, c0 + h, t, reinterpret_cast<float*>(v) + h);
                if (h16) sum_partials(part, G, G.n_a, 1, c0 + h, t, reinterpret_cast<float*>(up) + h);
            }
        } else {
            if constexpr (CH == 32) {
                tmem_ld32_async(taddr + (uint32_t)c0, v);
                if (h16) tmem_ld32_async(taddr + (uint32_t)(bn + c0), up);
            } else {
                tmem_ld16_async(taddr + (uint32_t)c0, v);
                if (h16) tmem_ld16_async(taddr + (uint32_t)(bn + c0), up);
            }
            tmem_wait_ld();
        }
        if (slot == 0) {   // the copies out of the slots (of the last unit, or of the last round) have read them
            if (elect_one()) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            __syncwarp();
        }
        uint8_t* const sl = base + (uint32_t)slot * slot_bytes;
        if (h16) {
#pragma unroll
            for (int c = 0; c < CH; ++c)
                *reinterpret_cast<bf16*>(sl + (lane >> 4) * (CH * 32) + c * 32 + (lane & 15) * 2) =
                    from_f<bf16>(silu_f(__uint_as_float(v[c])) * __uint_as_float(up[c]));
        } else {
#pragma unroll
            for (int c = 0; c < CH; ++c)
                *reinterpret_cast<uint32_t*>(sl + c * 128 + (((lane >> 2) ^ (c & 7)) << 4) + (lane & 3) * 4) = v[c];
        }
        const int tok0 = x.tok_tile * bn + c0;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (n0 < args.ep.n && tok0 < args.ep.m_tok && elect_one()) {
            if (mode == OUT_ADD) {
                tma_reduce(&args.map_o, smem_u32(sl), n0, tok0, 0);
            } else if (mode == OUT_F32) {
                tma_store(&args.map_o, smem_u32(sl), n0, tok0, 0);
            } else {
                tma_store(&args.map_o, smem_u32(sl), n0, tok0, 0);
                if (nw > 16 && n0 + 16 < args.ep.n) tma_store(&args.map_o, smem_u32(sl) + CH * 32, n0 + 16, tok0, 0);
            }
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
        if (++slot == args.n_slots) slot = 0;
    }
}

// kAux = false: the projections of the draft step (every activation group belongs to its weight
// group; the epilogues without bias). kAux = true adds the activation addressing of the fusion
// variants (a shared activation group, a contraction across stacked groups) and the biased store;
// it is a separate instance so that the draft step's code is not touched by it.
template <bool kAux>
__global__ void __launch_bounds__(kThreads, 1) gemm_tc_kernel(const __grid_constant__ TcArgs args) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t pad = (1024u - (raw & 1023u)) & 1023u;
    uint8_t* smem = smem_raw + pad;
    const uint32_t sbase = raw + pad;
    Geom G;
    G.n_units = args.n_units;
    G.n_tiles = args.n_tiles;
    G.tok_tiles = args.tok_tiles;
    G.splits = args.splits;
    G.kb_per_split = args.kb_per_split;
    G.k_blocks = args.k_blocks;
    G.n_a = args.n_a;
    G.kbs = args.kbs;
    G.bn = args.bn;
    G.n_bufs = args.n_bufs;
    G.pair = args.pair;
    G.a_bytes = args.a_bytes;
    G.b_bytes = args.b_bytes;
    G.stage_bytes = args.stage_bytes;
    G.idesc = args.idesc;
    uint32_t* const err = args.err;
    const int S = args.stages;
    float* epi = reinterpret_cast<float*>(smem + (size_t)S * G.stage_bytes);
    uint64_t* bars = reinterpret_cast<uint64_t*>(reinterpret_cast<uint8_t*>(epi) + args.epi_bytes);
    uint32_t* misc = reinterpret_cast<uint32_t*>(bars + 2 * S + 5);
    const uint32_t bar0 = smem_u32(bars);
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (S + s); };
    auto tfull_bar = [&](int b) { return bar0 + 8u * (2 * S + b); };
    auto tempty_bar = [&](int b) { return bar0 + 8u * (2 * S + 2 + b); };
    const uint32_t drain_bar = bar0 + 8u * (2 * S + 4);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned long long* const tst = args.t_stamps;
    if (tst && threadIdx.x == 0) atomicMin(tst, (unsigned long long)globaltimer_ns());
    if (warp == 4 && lane == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&args.map_a)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&args.map_b)) : "memory");
        if (args.out_mode != OUT_REGS)
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&args.map_o)) : "memory");
        if (G.n_a == 2)
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&args.map_a2)) : "memory");
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(full_bar(s), 1);
            mbar_init(empty_bar(s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(tfull_bar(b), 1);
            mbar_init(tempty_bar(b), 128);
        }
        mbar_init(drain_bar, 1);
        misc[1] = 0;
        misc[2] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 5) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&misc[0])),
                     "r"(args.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = misc[0];
    volatile int* abort_flag = reinterpret_cast<volatile int*>(&misc[1]);
    const int acc_cols = G.n_a * G.bn;

    if (warp == 4) {
        if (elect_one()) {
            // ---------------- TMA producer
            const CUtensorMap* mA = &args.map_a;
            const CUtensorMap* mA2 = &args.map_a2;
            const CUtensorMap* mB = &args.map_b;
            int stage = 0;
            uint32_t phase = 0, issued = 0, issued_phase = 0;
            bool ok = true;
            uint64_t policy = 0;
            asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
            const uint32_t b_base = G.a_bytes * G.n_a * G.kbs;
            const uint32_t tx = G.a_bytes * G.n_a + G.b_bytes;
            // first weight row of a unit in both maps (a pair's second map starts 128 rows in)
            const int row_step = args.bm << G.pair;
            // Weights do not depend on the previous kernel: the first ring of stages gets its
            // weight tiles before griddepcontrol.wait, the activation tiles after it.
            int pend_kx[kMaxStages], pend_nk[kMaxStages], pend_tok[kMaxStages], pend_grp[kMaxStages];
            uint32_t pend_st[kMaxStages];
            int npend = 0;
            bool waited = false;
            auto load_b = [&](uint32_t st, int kx0, int nk, int tok_tile, int group, uint32_t bar) {
                if constexpr (kAux) {
                    for (int j = 0; j < nk; ++j) {
                        int bx = kx0 + j * kBK, bz = group * args.b_gsel;
                        if (args.b_kg > 0) {   // contraction over stacked activation groups (Eq. 1)
                            bz = bx / args.b_kg;
                            bx -= bz * args.b_kg;
                        }
                        tma_load_3d(st + b_base + j * G.b_bytes, mB, bx, tok_tile * G.bn, bz, bar);
                    }
                } else {
                    for (int j = 0; j < nk; ++j)
                        tma_load_3d(st + b_base + j * G.b_bytes, mB, kx0 + j * kBK, tok_tile * G.bn, group, bar);
                }
            };
            for (int u = blockIdx.x; u < G.n_units && ok; u += gridDim.x) {
                const Unit x = decode_unit(G, u);
                for (int kb = x.kb0; kb < x.kb1; kb += G.kbs) {
                    const int nk = min(G.kbs, x.kb1 - kb);
                    if (!bar_wait(empty_bar(stage), phase ^ 1u, abort_flag, err)) {
                        ok = false;
                        break;
                    }
                    const uint32_t st = sbase + (uint32_t)stage * G.stage_bytes;
                    mbar_expect_tx(full_bar(stage), (uint32_t)nk * tx);
                    for (int j = 0; j < nk; ++j) {
                        const int kx = (kb + j) * kBK;
                        tma_load_3d_hint(st + j * G.a_bytes, mA, kx, x.n_tile * row_step, x.group, full_bar(stage), policy);
                        if (G.n_a == 2)
                            tma_load_3d_hint(st + (G.kbs + j) * G.a_bytes, mA2, kx, x.n_tile * row_step, x.group,
                                             full_bar(stage), policy);
                    }
                    if (waited) {
                        load_b(st, kb * kBK, nk, x.tok_tile, x.group, full_bar(stage));
                    } else {
                        pend_kx[npend] = kb * kBK;
                        pend_nk[npend] = nk;
                        pend_tok[npend] = x.tok_tile;
                        pend_grp[npend] = x.group;
                        pend_st[npend] = (uint32_t)stage;
                        if (++npend == S) {
                            pdl_wait();
                            if (tst) atomicMin(tst + args.t_slots, (unsigned long long)globaltimer_ns());
                            waited = true;
                            for (int i = 0; i < npend; ++i)
                                load_b(sbase + pend_st[i] * G.stage_bytes, pend_kx[i], pend_nk[i],
                                       pend_tok[i], pend_grp[i], full_bar(pend_st[i]));
                        }
                    }
                    issued |= 1u << stage;
                    issued_phase = (issued_phase & ~(1u << stage)) | (phase << stage);
                    if (++stage == S) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
            }
            if (!waited) {
                pdl_wait();
                if (tst) atomicMin(tst + args.t_slots, (unsigned long long)globaltimer_ns());
                for (int i = 0; i < npend; ++i)
                    load_b(sbase + pend_st[i] * G.stage_bytes, pend_kx[i], pend_nk[i], pend_tok[i],
                           pend_grp[i], full_bar(pend_st[i]));
            }
            // no copy is still landing in shared memory when the CTA exits, after a timeout either
            for (int s = 0; s < S; ++s)
                if (issued & (1u << s)) {
                    volatile int never = 0;
                    bar_wait(full_bar(s), (issued_phase >> s) & 1u, &never, err);
                }
        }
    } else if (warp == 5) {
        if (elect_one()) {
            // ---------------- MMA issuer
            int stage = 0, acc = 0;
            uint32_t phase = 0, acc_phase = 0;
            bool ok = true;
            const uint32_t b_base = G.a_bytes * G.n_a * G.kbs;
            for (int u = blockIdx.x; u < G.n_units && ok; u += gridDim.x) {
                const Unit x = decode_unit(G, u);
                if (!bar_wait(tempty_bar(acc), acc_phase ^ 1u, abort_flag, err)) break;
                tc_fence_after();
                const uint32_t d0 = tmem + (uint32_t)(acc * acc_cols);
                for (int kb = x.kb0; kb < x.kb1; kb += G.kbs) {
                    const int nk = min(G.kbs, x.kb1 - kb);
                    if (!bar_wait(full_bar(stage), phase, abort_flag, err)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t st = sbase + (uint32_t)stage * G.stage_bytes;
                    for (int j = 0; j < nk; ++j) {
                        const uint64_t da = smem_desc(st + j * G.a_bytes);
                        const uint64_t da2 = smem_desc(st + (G.kbs + j) * G.a_bytes);
                        const uint64_t db = smem_desc(st + b_base + j * G.b_bytes);
#pragma unroll
                        for (int k = 0; k < kBK / 16; ++k) {
                            const uint32_t accum = (kb > x.kb0 || j > 0 || k > 0) ? 1u : 0u;
                            umma_bf16(d0, da + 2 * k, db + 2 * k, G.idesc, accum);
                            if (G.n_a == 2) umma_bf16(d0 + G.bn, da2 + 2 * k, db + 2 * k, G.idesc, accum);
                        }
                    }
                    umma_commit(empty_bar(stage));
                    if (++stage == S) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
                if (!ok) break;
                umma_commit(tfull_bar(acc));
                if (G.n_bufs == 2) {
                    acc ^= 1;
                    if (acc == 0) acc_phase ^= 1u;
                } else {
                    acc_phase ^= 1u;
                }
            }
            // all issued MMAs complete before TMEM is released
            umma_commit(drain_bar);
            volatile int never = 0;
            bar_wait(drain_bar, 0, &never, err);
        }
    } else {
        // ---------------- epilogue warps 0-3 (thread t <-> TMEM lane t <-> feature t of a tile)
        pdl_wait();
        // dependents may start once every CTA has passed its own dependency wait: everything the
        // kernels before this one wrote is then complete (the attention that follows the Q/K^d/V^d
        // projection reads the context cache before its own wait)
        if (threadIdx.x == 0) pdl_trigger();
        const int t = threadIdx.x;
        int acc = 0;
        uint32_t acc_phase = 0;
        const int bn = G.bn, na = G.n_a;
        float* const ws = args.ws;
        const int mode = args.out_mode;
        const bool resid = args.ep.kind == EPI_RESID && bn == kChunk && mode == OUT_REGS;
        for (int u = blockIdx.x; u < G.n_units; u += gridDim.x) {
            const Unit x = decode_unit(G, u);
            if (mode != OUT_REGS) {
                const bool got = bar_wait(tfull_bar(acc), acc_phase, abort_flag, err);
                if (!__all_sync(0xffffffffu, got)) break;
                tc_fence_after();
                const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(acc * acc_cols);
                const float* part = nullptr;   // K splits through the workspace: this tile's partials
                bool mine = true;
                if (mode != OUT_ADD && G.splits > 1) {
                    mine = split_partials(args, G, x, taddr, tempty_bar(acc), misc, t);
                    part = ws + (size_t)x.tile_id * G.splits * na * bn * 128;
                }
                if (mine) {
                    if (bn % 32 == 0)
                        staged_out<32>(args, G, x, taddr, part, epi, warp, lane);
                    else
                        staged_out<16>(args, G, x, taddr, part, epi, warp, lane);
                }
                if (!part) {
                    tc_fence_before();
                    mbar_arrive(tempty_bar(acc));
                }
                if (G.n_bufs == 2) {
                    acc ^= 1;
                    if (acc == 0) acc_phase ^= 1u;
                } else {
                    acc_phase ^= 1u;
                }
                continue;
            }
            // the residual rows do not depend on the accumulator: load them before waiting
            float rr[kChunk];
            if (resid) load_resid(args.ep, x.n_tile, x.tok_tile * bn, t, rr);
            if (!bar_wait(tfull_bar(acc), acc_phase, abort_flag, err)) break;
            tc_fence_after();
            const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(acc * acc_cols);
            bool final_tile = true;
            if (G.splits > 1) final_tile = split_partials(args, G, x, taddr, tempty_bar(acc), misc, t);
            if (final_tile) {
                for (int c0 = 0; c0 < bn; c0 += kChunk) {
                    for (int a = 0; a < na; ++a) {
                        float v[kChunk];
                        if (G.splits == 1) {
                            tmem_ld16(taddr + (uint32_t)(a * bn + c0), v);
                        } else {
                            sum_partials(ws + (size_t)x.tile_id * G.splits * na * bn * 128, G, na, a, c0, t, v);
                        }
#pragma unroll
                        for (int c = 0; c < kChunk; ++c) epi[(a * kChunk + c) * 128 + t] = v[c];
                    }
                    epi_bar();
                    if (resid)
                        resid_epilogue(args.ep, epi, x.n_tile, x.tok_tile * bn + c0, t, rr);
                    else if (G.pair)   // two 128-feature tiles, one per accumulator
                        for (int a = 0; a < 2; ++a)
                            apply_epilogue<bf16, kAux>(args.ep, epi + a * kChunk * 128, x.group,
                                                       2 * x.n_tile + a, x.tok_tile * bn + c0, t);
                    else
                        apply_epilogue<bf16, kAux>(args.ep, epi, x.group, x.n_tile, x.tok_tile * bn + c0, t);
                    epi_bar();
                }
            }
            if (G.splits == 1) {
                tc_fence_before();
                mbar_arrive(tempty_bar(acc));
            }
            if (G.n_bufs == 2) {
                acc ^= 1;
                if (acc == 0) acc_phase ^= 1u;
            } else {
                acc_phase ^= 1u;
            }
        }
        // the copies have read the staging slots before the CTA's shared memory goes (what they write is
        // visible to the dependents with the end of the grid, as any store's)
        if (mode != OUT_REGS) {
            __syncwarp();
            if (elect_one()) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        }
    }
    __syncthreads();
    if (tst && threadIdx.x == 0) atomicMax(tst + 2 * args.t_slots, (unsigned long long)globaltimer_ns());
    if (warp == 5) {
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(args.tmem_cols)
                     : "memory");
    }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                             &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

// bf16 tensor [groups][rows][k] (row stride k, group stride group_rows rows) -> 3-D tensor map
// with a box of 64 (k) x box_rows x 1, 128-byte swizzle, zero fill outside the tensor.
bool make_map(CUtensorMap* m, const void* base, int k, int rows, int groups, long long group_rows,
              int box_rows) {
    auto enc = encode_fn();
    if (!enc) return false;
    cuuint64_t dims[3] = {(cuuint64_t)k, (cuuint64_t)rows, (cuuint64_t)groups};
    cuuint64_t strides[2] = {(cuuint64_t)k * 2, (cuuint64_t)group_rows * k * 2};
    cuuint32_t box[3] = {(cuuint32_t)kBK, (cuuint32_t)box_rows, 1};
    cuuint32_t es[3] = {1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box,
               es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

static bool encode_tma(CUtensorMap* m, CUtensorMapDataType type, const void* base, int rank,
                       const uint64_t* dims, const uint64_t* strides_bytes, const uint32_t* box,
                       CUtensorMapSwizzle swizzle = CU_TENSOR_MAP_SWIZZLE_128B) {
    auto enc = encode_fn();
    if (!enc || rank < 1 || rank > 5) return false;
    cuuint64_t d[5], st[4];
    cuuint32_t bx[5], es[5];
    for (int i = 0; i < rank; ++i) {
        d[i] = dims[i];
        bx[i] = box[i];
        es[i] = 1;
        if (i + 1 < rank) st[i] = strides_bytes[i];
    }
    return enc(m, type, (cuuint32_t)rank, const_cast<void*>(base), d, st, bx, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
bool encode_tma_bf16(CUtensorMap* m, const void* base, int rank, const uint64_t* dims,
                     const uint64_t* strides_bytes, const uint32_t* box) {
    return encode_tma(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, base, rank, dims, strides_bytes, box);
}
// packed boxes (no swizzle)
static bool encode_tma_packed(CUtensorMap* m, const void* base, const uint64_t* dims, const uint64_t* strides_bytes,
                              const uint32_t* box) {
    return encode_tma(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, base, 3, dims, strides_bytes, box, CU_TENSOR_MAP_SWIZZLE_NONE);
}
bool encode_tma_f32(CUtensorMap* m, const void* base, int rank, const uint64_t* dims,
                    const uint64_t* strides_bytes, const uint32_t* box) {
    return encode_tma(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, base, rank, dims, strides_bytes, box);
}

cudaError_t launch_gemm_tc(dflare_ctx* c, const GemmDesc& g, cudaStream_t s, std::string* why) {
    if (g.m_tok <= 0 || g.n <= 0) return cudaSuccess;
    TcArgs a;
    memset(&a, 0, sizeof(a));
    a.bn = g.m_tok <= 256 ? ((g.m_tok + 15) / 16) * 16 : 256;
    // A projection with few weight tiles is divided over the SMs by tokens (tiles of 64 rows at
    // least) before it is divided along K, where K splits would go through the workspace: at 240
    // tokens each split writes 120 KB of partials and the last CTA of a tile reads all of them
    // back, while token tiles only read the weights again from L2. LM head of 4096 entries, d 4096:
    // one layer with 240 such rows 237.1 -> 224.8 us, with 248 rows and long contexts 373.7 ->
    // 353.4 us (4 K splits of a 256-token tile against 4 tiles of 64).
    const bool ws_splits = g.ep.kind != EPI_RED32 && !(g.ep.kind == EPI_RESID && !(c->cfg.flags & DFLARE_FLAG_DETERMINISTIC));
    const long long w_tiles = (long long)g.groups * ((g.n + kBM - 1) / kBM);
    // (DFlash's FC keeps K splits: its contraction of T d is long enough to outweigh the partials)
    while (ws_splits && g.b_kgroup == 0 && a.bn >= 128 &&
           w_tiles * ((g.m_tok + a.bn / 2 - 1) / (a.bn / 2)) <= c->num_sms)
        a.bn = (a.bn / 2 + 15) / 16 * 16;
    // With token tiles of 128 or more rows the GEMM is bound by the tensor pipeline, not by HBM:
    // two adjacent 128-row weight tiles can then share one activation tile (two accumulators, as
    // the SwiGLU gate and up tiles do), a third fewer shared-memory bytes per FLOP. At 256 token
    // rows the pair fills all 512 TMEM columns, so a unit's epilogue no longer overlaps the next
    // unit's MMAs: pairs pay only for the cheap fp32-logit epilogue (the LM head), and only when
    // their wave count times ~1.8 single-tile units beats the single tiles' wave count (batch-16
    // step 1.965 -> 1.947 ms). The two-SM GEMM has taken heads of more than 160 rows over; pairs remain for large
    // heads of 113 to 160 rows and for vocabularies whose rows do not start on 16 bytes. Measured at 120 / 135 /
    // 150 rows of 151936 entries, d 4096 (us): pairs 207 / 219 / 224, single tiles of 64 to 128 rows 207 / 210 / 219,
    // two-SM 220 / 221 / 223; 120 / 150 rows of 201088 entries, d 2880: 213 / 246, 221 / 244, 222 / 226; 120 rows of
    // 32000 entries, d 2560: 34 / 32 / 37. None of the three leads throughout.
    {
        const long long u1 = (long long)g.groups * ((g.n + kBM - 1) / kBM) * ((g.m_tok + a.bn - 1) / a.bn);
        const long long u2 = (long long)g.groups * ((g.n + 2 * kBM - 1) / (2 * kBM)) * ((g.m_tok + a.bn - 1) / a.bn);
        const long long w1 = (u1 + c->num_sms - 1) / c->num_sms, w2 = (u2 + c->num_sms - 1) / c->num_sms;
        a.pair = (!g.a2 && a.bn >= 128 && g.n > kBM &&
                  g.ep.kind == EPI_F32 && 9 * w2 < 5 * w1) ? 1 : 0;
    }
    a.n_a = (g.a2 || a.pair) ? 2 : 1;
    a.tok_tiles = (g.m_tok + a.bn - 1) / a.bn;
    // SwiGLU and logit tiles of fewer weight rows where that divides the waves better: its K splits would go through
    // the workspace, and 128-row tiles leave a third of the SMs without any weights to stream (d 4096, ffn
    // 12288: 96 tiles of 128, 128 of 96). The MMA still multiplies 128 rows; those past the tile's (whatever
    // lies behind it in shared memory) end in accumulator lanes that nobody reads. One launch, 128-row tiles
    // -> these: 64 tokens, d 4096 (128 tiles of 96) 34.4 -> 33.3 us; 16 tokens, d 2560 (152 of 64, no K splits)
    // 19.6 -> 18.0; 32 tokens, GPT-OSS (144 of 80) 24.3 -> 22.1. Likewise for logits, in steps of 32 rows: 40000
    // entries (417 tiles of 96 in 3 waves instead of 313 of 128) at 48 tokens 62.6 -> 53.4.
    a.bm = kBM;
    const bool swiglu_tma = g.ep.kind == EPI_SWIGLU && (reinterpret_cast<uintptr_t>(g.ep.out) & 15u) == 0 && g.ep.ldo % 8 == 0;
    const bool f32_tma = g.ep.kind == EPI_F32 && !a.pair && (reinterpret_cast<uintptr_t>(g.ep.out) & 15u) == 0 && g.ep.ldo % 4 == 0;
    if (swiglu_tma || f32_tma) {
        // A gate/up tile counts four rows more for its hand-overs. A logit tile of bn tokens counts bn^2 / 160 more, and
        // 64 rows are taken only where one wave holds them all: at few tokens its weights' stream covers the rest, at
        // many the tokens' own stream and the multiplication of 128 rows do not shrink with it. Measured (d 4096, us of
        // tiles of 128 / 96 / 64 rows): 65024 entries (4 / 5 / 7 waves) 30 tokens 84.5 / 80.6 / 82.5, 60 tokens
        // 86.7 / 88.9 / 107.6, 105 tokens 95.1 / 101.5 / 125.9; 128256 (7 / 9 / 14) 30 tokens 157.7 / 151.0 / 161.7, 60
        // 158.2 / 161.2 / 212.8, 105 174.4 / 185.6 / 247.5; 100352 (6 / 7 / 11) 60 131.5 / 126.5 / 167.7. Over ten
        // vocabularies, three widths and 15 to 105 tokens the choice is 4 % behind the best of the three at most, but for
        // 65024 entries at d 2048 and 60 tokens (8 %).
        long long best_cost = 0;
        for (int bm = kBM; bm >= 64; bm -= swiglu_tma ? 16 : 32) {
            const long long t = (long long)g.groups * ((g.n + bm - 1) / bm) * a.tok_tiles;
            const long long waves = (t + c->num_sms - 1) / c->num_sms;
            if (!swiglu_tma && bm == 64 && waves > 1) continue;
            const long long cost = waves * (160 * bm + (swiglu_tma ? 160 * 4 : a.bn * a.bn));
            if (bm == kBM || cost < best_cost) {
                best_cost = cost;
                a.bm = bm;
            }
        }
    }
    a.n_tiles = (g.n + (a.bm << a.pair) - 1) / (a.bm << a.pair);
    a.k_blocks = (g.k + kBK - 1) / kBK;
    const int tiles = g.groups * a.n_tiles * a.tok_tiles;
    const int sms = c->num_sms;
    // split-K choice: the most splits that still run as one wave (tiles * splits <= SMs), within
    // the workspace and counter capacity. Measured: a second wave of split units is slower than
    // fewer, longer units even when it shortens every unit (d 4096 gate/up: 3 splits over 288
    // units 97 us, 1 split over 96 units 42 us), so no split count that spills into a second
    // wave is taken.
    int best = 1;
    for (int sp = 2; sp <= 16 && sp <= a.k_blocks / 2 && tiles * sp <= sms; ++sp) {
        const int kbp = (a.k_blocks + sp - 1) / sp;
        const int spn = (a.k_blocks + kbp - 1) / kbp;
        const size_t need = (size_t)tiles * spn * a.n_a * a.bn * 128;
        if (need > c->ws_floats || tiles > c->tile_cnt_n) break;
        best = spn;
    }
    // Shared-memory budget: up to 227 KB (one CTA per SM; measured faster than two smaller CTAs
    // per SM, with or without programmatic dependent launch).
    // results through TMA where every row of the output starts on 16 bytes (and no pair of tiles is formed)
    const bool det = c->cfg.flags & DFLARE_FLAG_DETERMINISTIC;
    auto rows16 = [](const void* p, long long ld_bytes) {
        return (reinterpret_cast<uintptr_t>(p) & 15u) == 0 && ld_bytes % 16 == 0;
    };
    if (g.ep.kind == EPI_RED32) {
        if (!rows16(g.ep.out, 4ll * g.ep.ldo)) {
            if (why) *why = "tcgen05 GEMM: fp32 sums need 16-byte aligned rows";
            return cudaErrorInvalidValue;
        }
        a.out_mode = OUT_ADD;
    }
    if (g.ep.kind == EPI_RESID && !det && rows16(g.ep.resid, 4ll * g.ep.ld_resid)) a.out_mode = OUT_ADD;
    if (swiglu_tma) a.out_mode = OUT_SWIGLU;
    if (f32_tma) a.out_mode = OUT_F32;
    const int ch = a.bn % 32 == 0 ? 32 : 16;   // tokens per staging slot
    const int kb_bytes = a.bm * kBK * 2 * a.n_a + a.bn * kBK * 2;   // one k-block of a stage
    const int misc_bytes = 16;
    // (128-row operand reads that start at a shorter tile end inside the allocation)
    const int slack = (kBM - a.bm) * kBK * 2;
    auto epi_of = [&](int slots) {
        return a.out_mode == OUT_REGS ? a.n_a * kChunk * 128 * 4 : 4 * slots * ch * (a.out_mode == OUT_SWIGLU ? 64 : 128);
    };
    auto fixed_of = [&](int slots) { return 1024 + epi_of(slots) + 8 * (2 * kMaxStages + 5) + misc_bytes + slack; };
    // staging for 64 tokens; for 32 where only that leaves room for a third stage of two k-blocks. One launch,
    // 64 -> 32: 144 tokens, d 4096: O 12.7 -> 11.1 us, down 22.9 -> 21.8; 155 logit rows of 40000 entries 74.2 -> 68.3.
    // (Where the ring stays the same, 32 cost up to 0.5 us: Q/K/V at 160 tokens 13.3 -> 13.7.)
    a.n_slots = std::min(a.bn / ch, 64 / ch);
    if (6 * kb_bytes > kSmemLimit - fixed_of(a.n_slots) && 6 * kb_bytes <= kSmemLimit - fixed_of(32 / ch)) a.n_slots = 32 / ch;
    const int epi_bytes = epi_of(a.n_slots), fixed = fixed_of(a.n_slots);
    a.epi_bytes = epi_bytes;
    // a hand-off costs about 300 clocks whatever its bytes, and a ring of two stages runs dry: four
    // 64-wide k-blocks a stage where three stages fit, else two where three fit, else one. Measured (us
    // after the dependency at 4 / 2 / 1): 64 tokens, d 4096: Q/K/V 11.7 / 11.5 / 12.4, down 20.0 / 19.1 / 21.0; 96
    // tokens Q/K/V - / 11.9 / 12.8, down - / 20.1 / 22.0, LM head of 40000 entries - / 59.4 / 72.4; 16 tokens, d 2560:
    // O 5.8 / 6.2 / 7.3. Gate/up at 2 / 1: 16 tokens, d 4096, ffn 16384 41.6 / 43.9, d 2560, ffn 19456 30.5 / 31.7; 32
    // tokens 31.6 / 33.3; 64 tokens, d 4096, ffn 12288 34.4 / 35.1, d 2880, ffn 11520 23.6 / 24.3; 96 tokens, d 2560,
    // ffn 9728 19.8 / 22.0.
    a.kbs = 3 * 4 * kb_bytes <= kSmemLimit - fixed ? 4 : 3 * 2 * kb_bytes <= kSmemLimit - fixed ? 2 : 1;
    a.kb_per_split = (a.k_blocks + best - 1) / best;
    // (split ranges are not rounded to whole stages: the producer issues a partial last stage,
    // and balanced ranges beat 512-byte-aligned ones, e.g. Q/K^d/V^d 14/14/12 k-blocks rather
    // than 16/16/8: 0.5265 -> 0.5221 ms per Qwen3-4B-shaped step)
    a.splits = (a.k_blocks + a.kb_per_split - 1) / a.kb_per_split;
    if (a.splits > 1 && ((size_t)tiles * a.splits * a.n_a * a.bn * 128 > c->ws_floats || tiles > c->tile_cnt_n)) {
        if (why) *why = "tcgen05 GEMM: split-K workspace too small";
        return cudaErrorInvalidValue;
    }
    a.n_units = tiles * a.splits;
    a.b_bytes = (uint32_t)a.bn * kBK * 2;
    a.a_bytes = (uint32_t)a.bm * kBK * 2;
    a.stage_bytes = (uint32_t)a.kbs * (a.a_bytes * a.n_a + a.b_bytes);
    a.stages = std::min(kMaxStages, (kSmemLimit - fixed) / (int)a.stage_bytes);
    if (a.stages < 2) {
        if (why) *why = "tcgen05 GEMM: tile does not fit in shared memory";
        return cudaErrorInvalidValue;
    }
    const int smem = 1024 + a.stages * (int)a.stage_bytes + epi_bytes + 8 * (2 * a.stages + 5) + misc_bytes + slack;
    a.n_bufs = (2 * a.n_a * a.bn <= 512) ? 2 : 1;
    int cols = 32;
    while (cols < a.n_bufs * a.n_a * a.bn) cols <<= 1;
    a.tmem_cols = cols;
    // kind::f16 instruction descriptor: fp32 accumulate, bf16 A and B, both K-major,
    // N = bn (bits 17-22, N >> 3), M = 128 (bits 24-28, M >> 4)
    a.idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(a.bn >> 3) << 17) |
              ((uint32_t)(kBM >> 4) << 24);
    a.ws = c->ws;
    a.tile_cnt = c->tile_cnt;
    a.err = c->err;
    a.ep = g.ep;
    // weights: groups of n rows, a_group_rows apart; activations: one group per weight group, one
    // group shared by all (b_shared), or k / b_kgroup groups that the contraction runs across
    const long long a_gr = g.a_group_rows > 0 ? g.a_group_rows : g.n;
    a.b_kg = g.b_kgroup;
    a.b_gsel = g.b_shared ? 0 : 1;
    const int b_k = g.b_kgroup > 0 ? g.b_kgroup : g.k;
    const int b_groups = g.b_kgroup > 0 ? g.k / g.b_kgroup : (g.b_shared ? 1 : g.groups);
    const long long b_gr = g.b_group_rows > 0 ? g.b_group_rows : g.m_tok;
    if (g.b_kgroup > 0 && (g.b_kgroup % kBK != 0 || g.k % g.b_kgroup != 0 || g.groups != 1)) {
        if (why) *why = "tcgen05 GEMM: b_kgroup must be a multiple of 64 that divides k, with one group";
        return cudaErrorInvalidValue;
    }
    // a pair's second tile: the same matrix from row 128 on (rows past its end read as zeros)
    const void* a2 = g.a2 ? g.a2 : a.pair ? static_cast<const void*>(static_cast<const bf16*>(g.a) + (size_t)kBM * g.k)
                                          : g.a;
    if (!make_map(&a.map_a, g.a, g.k, g.n, g.groups, a_gr, a.bm) ||
        !make_map(&a.map_a2, a2, g.k, a.pair ? g.n - kBM : g.n, g.groups, a_gr, a.bm) ||
        !make_map(&a.map_b, g.b, b_k, g.m_tok, b_groups, b_gr, a.bn)) {
        if (why) *why = "cuTensorMapEncodeTiled failed (alignment or driver entry point)";
        return cudaErrorInvalidValue;
    }
    if (a.out_mode != OUT_REGS) {
        const bool h16 = a.out_mode == OUT_SWIGLU;
        const uint64_t ld = h16 ? 2ull * g.ep.ldo : 4ull * (g.ep.kind == EPI_RESID ? g.ep.ld_resid : g.ep.ldo);
        const uint64_t dims[3] = {(uint64_t)g.n, (uint64_t)g.m_tok, 1}, st[2] = {ld, ld * (uint64_t)g.m_tok};
        const uint32_t box[3] = {h16 ? 16u : 32u, (uint32_t)ch, 1};
        void* out = g.ep.kind == EPI_RESID ? static_cast<void*>(g.ep.resid) : g.ep.out;
        if (!(h16 ? encode_tma_packed(&a.map_o, out, dims, st, box) : encode_tma_f32(&a.map_o, out, 3, dims, st, box))) {
            if (why) *why = "cuTensorMapEncodeTiled failed (output)";
            return cudaErrorInvalidValue;
        }
    }
    const bool aux = g.b_kgroup > 0 || g.b_shared || g.ep.bias || g.ep.out_gstride;
    static PerDeviceOnce configured[2];
    const cudaError_t ce = configured[aux]([aux] {
        return cudaFuncSetAttribute(aux ? gemm_tc_kernel<true> : gemm_tc_kernel<false>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
    });
    if (ce != cudaSuccess) return ce;
    const int grid = std::min(a.n_units, sms);
    if (c->t_stamps && c->t_next < c->t_slots) {
        a.t_stamps = c->t_stamps + c->t_next++;
        a.t_slots = c->t_slots;
    }
    return launch_kernel(c->pdl, aux ? gemm_tc_kernel<true> : gemm_tc_kernel<false>, dim3(grid),
                         dim3(kThreads), smem, s, a);
}

}  // namespace dfl
