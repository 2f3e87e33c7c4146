// Token-level state access on tensor cores (bf16 I/O, D = 128): the comparison mode of the paper's
// "State access granularity" ablation (Sec. 4.3).  Token i of the block reads the state advanced by the
// block's tokens before it,
//   S^(0) = S,  S^(i+1) = alpha_i S^(i) + K'_i^T V'_i,   X_i = Q'_i S^(i),
// which is a causal linear attention over the block on top of the carried state.  This kernel ADDS
// sigmoid(g_i) X_i to an output that already holds the intra-block softmax branch; S is only read.
//
// Chunkwise form (own derivation), chunks of C = 128 tokens, inside a chunk that enters with state
// S_c:  lg_j = sum_{m <= j} log alpha_m,  la_i = lg_{i-1} (la_0 = 0),  w_j = exp(lg_last - lg_j) <= 1,
//   Khat_j = w_j K'_j,   Shat = exp(lg_last) S_c,
//   X_i = exp(la_i - lg_last) [ Q'_i Shat + sum_{j < i} (Q'_i . Khat_j) V'_j ],
//   S_{c+1} = Shat + Khat^T V'.
// Every factor that multiplies an operand is <= 1; only the final row factor exp(la_i - lg_last) is
// >= 1 (bounded by 1 / prod of the chunk's gates: gates that stay below about 0.5 for a whole chunk
// would leave the fp32 range, which a forget gate of a model that remembers anything never does).
//
// The chunks of a head depend on one another only through S_c, and what a stretch of chunks adds to the state
// is the commit's sum with the stretch's own decay weights.  So the flattened sequence of tiles is cut into the
// commit kernel's runs (one CTA each; a "segment" is what a run holds of one head) and four launches replace
// one CTA per head walking all its chunks (12 heads x 1560 tokens: 159 us on 12 SMs -> 56 us; 4680 tokens: 440 -> 75).
// Where heads are short the runs are whole heads and this kernel goes alone:
//   run_decay_weights   decay of every token to the end of its segment, total decay of the segment
//   tc_commit_kernel    sum over the segment of (w K')^T V
//   tc_run_prefix       the state at the start of every segment, in order
//   this kernel         walks the chunks of one run, starting each segment from its state
// One CTA (256 threads, two per token row) per run; the fp32 state lives in TMEM.  Per chunk:
//   U_q, U_k, U_v = Q W_q, K W_k, V W_v                      3 MMAs into TMEM
//   pass 1: gates (log-space scan), Q' , Khat, V' as bf16 over the raw tiles; Shat into TMEM and as a
//           bf16 operand copy
//   SC = Q' Khat^T,  O = Q' Shat                             2 MMAs
//   pass 2: P = strictly lower triangle of SC as bf16 into TMEM
//   O += P V',  S += Khat^T V'                               2 MMAs
//   epilogue: out_i += sigmoid(g_i) exp(la_i - lg_last) O_i
// Every wait is bounded; on expiry the CTA records ARL2_ERR_TIMEOUT and leaves through the common exit.
#include "tc_common.cuh"

namespace arl2 {

namespace {

constexpr int kTRThreads = 256;
constexpr int kTROffWq = 0, kTROffWk = kTileBytes, kTROffWv = 2 * kTileBytes;
constexpr int kTROffQ = 3 * kTileBytes, kTROffK = 4 * kTileBytes, kTROffV = 5 * kTileBytes;
constexpr int kTROffS = 6 * kTileBytes;                 // bf16 copy of Shat, [d][e]; then the tile's output rows
constexpr int kTROffBars = 7 * kTileBytes;
constexpr int kTROffGates = kTROffBars + 128;           // lg[128], then warp totals
constexpr int kTRSmemBytes = kTROffGates + 128 * 4 + 64 + 1024;

enum TRBar : int { kTRBarW = 0, kTRBarLoad, kTRBarU, kTRBarA, kTRBarB, kTRBarOut, kTRBarDrain, kTRNumBars };

struct TcReadoutParams {
    Shape s;
    const uint4* rope_h;
    const float* alpha;        // [B, L, H] forget-gate logits, or nullptr = 1
    const float* gate;         // [B, L, H] combine-gate logits
    const float* state;        // [B, H, 128, 128] fp32, read only
    const float* entry;        // [B * H, nslot, 128 x 128]: state at the start of each segment (slot layout of the commit),
                               // or nullptr: every run is a whole head and starts from `state`
    uint32_t* status;
    uint32_t spin_limit;
    int ntile;                 // 128-token tiles per (stream, head)
    int total_tiles, share;    // runs of `share` tiles over all heads' tiles
    int nslot;
};

__global__ void __launch_bounds__(kTRThreads, 1)
tc_token_readout_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                        const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_wq,
                        const __grid_constant__ CUtensorMap tm_wk, const __grid_constant__ CUtensorMap tm_wv,
                        const __grid_constant__ CUtensorMap tm_o,   // [B, L, H, 128], boxes of 32 rows: receives += sigmoid(g) X
                        const TcReadoutParams p)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                               ~static_cast<uintptr_t>(1023));
    const uint32_t smem_base = smem_u32(smem);
    const uint32_t bars = smem_base + kTROffBars;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + kTROffBars + kTRNumBars * 8);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + kTROffBars + kTRNumBars * 8 + 4);
    float* lg_s = reinterpret_cast<float*>(smem + kTROffGates);          // [128] inclusive log products
    float* wsum = lg_s + 128;                                            // [4] warp totals
    const Abort ab{abort_flag, p.status, p.spin_limit};

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int L = p.s.L, H = p.s.H;
    const int g_begin = (int)blockIdx.x * p.share, g_end = min(p.total_tiles, g_begin + p.share);

    if (tid == 0) {
        for (int i = 0; i < kTRNumBars; ++i) mbar_init(bars + 8 * i, 1);
        *abort_flag = 0;
        fence_barrier_init();
        fence_proxy_async_smem();
    }
    if (warp == 0) {
        tmem_alloc(smem_u32(tmem_slot), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    // two threads per row: warps w and w + 4 own the same 32 TMEM lanes and split the 128 columns
    const int r = (warp & 3) * 32 + lane;
    const int hf = warp >> 2;
    const uint32_t lane_base = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
    // TMEM columns: U_q, later SC | U_k, later O | U_v, later P | S
    constexpr uint32_t kColQ = 0, kColK = kTile, kColV = 2 * kTile, kColS = 3 * kTile;

    bool ok = true;
    if (tid == 0) {
        prefetch_tensormap(&tm_q);
        prefetch_tensormap(&tm_k);
        prefetch_tensormap(&tm_v);
    }
    // the three tiles of the tile with flattened index g
    auto load_tiles = [&](int g) {
        const int bh = g / p.ntile, row0 = (g - bh * p.ntile) * kTile;
        const uint32_t bar = bars + 8 * kTRBarLoad;
        mbar_expect_tx(bar, 3 * kTileBytes);
        const CUtensorMap* maps[3] = {&tm_q, &tm_k, &tm_v};
        for (int i = 0; i < 3; ++i) {
            tma_load_4d(smem_base + kTROffQ + i * kTileBytes, maps[i], bar, 0, bh % H, row0, bh / H);
            tma_load_4d(smem_base + kTROffQ + i * kTileBytes + kHalfBytes, maps[i], bar, 64, bh % H, row0, bh / H);
        }
    };
    auto load_maps = [&](int h) {
        const uint32_t bar = bars + 8 * kTRBarW;
        mbar_expect_tx(bar, 3 * kTileBytes);
        const CUtensorMap* maps[3] = {&tm_wq, &tm_wk, &tm_wv};
        for (int i = 0; i < 3; ++i) {
            tma_load_2d(smem_base + i * kTileBytes, maps[i], bar, 0, h * kTile);
            tma_load_2d(smem_base + i * kTileBytes + kHalfBytes, maps[i], bar, 64, h * kTile);
        }
    };
    int loads = 0, map_loads = 0, out_loads = 0;
    if (tid == 0) {
        load_maps(g_begin / p.ntile % H);
        load_tiles(g_begin);
        loads = map_loads = 1;
    }

    constexpr uint32_t kLboK = 1u << 16;
    constexpr uint32_t kLboMN = (uint32_t)(kHalfBytes >> 4) << 16;
    const uint32_t desc_hi = (uint32_t)(smem_desc_sw128(0, 0) >> 32);
    auto desc64 = [&](uint32_t lo) {
        uint64_t d;
        asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(desc_hi));
        return d;
    };
    constexpr uint32_t idesc_kk = idesc_bf16(kTile, kTile, 0, 0);   // both operands contraction-contiguous
    constexpr uint32_t idesc_kn = idesc_bf16(kTile, kTile, 0, 1);   // B rows = contraction index
    constexpr uint32_t idesc_nn = idesc_bf16(kTile, kTile, 1, 1);   // both operands row = contraction index
    auto koff_k = [](int ks) { return (uint32_t)(((ks >> 2) * kHalfBytes + (ks & 3) * 32) >> 4); };
    auto koff_n = [](int ks) { return (uint32_t)(ks * (2048 >> 4)); };
    auto lo_of = [&](int off, uint32_t lbo) { return ((smem_base + (uint32_t)off) >> 4) | lbo; };

    // The gates and the rotation table of a tile are asked for a tile ahead (the first ones here): behind the wait for the
    // tiles and the first MMAs, which keep warp 0, they held the whole CTA up (12 heads x 1560 tokens 67.7 -> 65.8 us per pass, 12 x 4680 221 -> 218).
    float alpha_logit = 0.0f, gate_logit = 0.0f;
    uint4 cs[8];
    auto fetch_row = [&](int g) {
        const int bhi = g / p.ntile, b = bhi / H, h = bhi - b * H, row = (g - bhi * p.ntile) * kTile + r;
        if (row < L) {
            const size_t gi = ((size_t)b * L + row) * H + h;
            gate_logit = p.gate[gi];
            if (hf == 0 && p.alpha != nullptr) alpha_logit = p.alpha[gi];
        }
        if (p.rope_h != nullptr) {
            const uint4* tab = p.rope_h + ((size_t)(row >> 5) * 16 + hf * 8) * 32 + (row & 31);
#pragma unroll
            for (int i = 0; i < 8; ++i) cs[i] = tab[i * 32];
        }
    };
    fetch_row(g_begin);
    bool alive = true;
    uint32_t segs = 0;   // segments begun
    for (int g = g_begin; g < g_end; ++g) {
        const int bhi = g / p.ntile, tl = g - bhi * p.ntile;
        const int b = bhi / H, h = bhi - b * H;
        const size_t bh = (size_t)bhi;
        const bool seg_first = g == g_begin || tl == 0;
        const bool seg_last = g + 1 == g_end || tl + 1 == p.ntile;   // nothing of this run reads the state after it
        const uint32_t par = (uint32_t)(g - g_begin) & 1u;
        const int row = tl * kTile + r;                // this thread's token
        if (seg_first) {
            // The maps, Q, K and V are of the caller, not of the kernel before; the states and the output are not.
            if (g == g_begin) grid_dependency_sync();
            // the segment's state (fp32) into TMEM: row d = r, this thread's 64 columns
            const bool whole = p.entry == nullptr;
            const float* src = whole ? p.state + (bh * kTile + r) * kTile + hf * 64
                                     : p.entry + (bh * p.nslot + (size_t)(blockIdx.x - (bhi * p.ntile) / p.share)) * kTile * kTile +
                                           ((size_t)(hf * 8) * kTile + r) * 8;
            const size_t step8 = whole ? 8 : (size_t)kTile * 8;   // from one group of 8 columns to the next
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                uint32_t x[32];
#pragma unroll
                for (int e = 0; e < 4; ++e)
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const float4 v = *reinterpret_cast<const float4*>(src + (size_t)(c * 4 + e) * step8 + q * 4);
                        x[e * 8 + q * 4 + 0] = __float_as_uint(v.x); x[e * 8 + q * 4 + 1] = __float_as_uint(v.y);
                        x[e * 8 + q * 4 + 2] = __float_as_uint(v.z); x[e * 8 + q * 4 + 3] = __float_as_uint(v.w);
                    }
                tmem_st32(lane_base + kColS + hf * 64 + c * 32, x);
            }
            tmem_wait_st();
            ++segs;
        }
        if (lane == 0) tma_store_wait_read();   // the last tile's rows have left the place where Shat goes
        // ---- gates of the chunk: lg_j = sum_{m <= j} log alpha_m (tokens past L: alpha = 1)
        float la_log = 0.0f;   // log alpha of this thread's token
        if (hf == 0) {
            if (row < L && p.alpha != nullptr) {
                const float x = alpha_logit;
                la_log = x >= 0.0f ? -log1pf(expf(-x)) : x - log1pf(expf(x));
            }
            float cl = la_log;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const float up = __shfl_up_sync(0xffffffffu, cl, off);
                if (lane >= off) cl += up;
            }
            if (lane == 31) wsum[warp] = cl;
            lg_s[r] = cl;              // within the warp so far
        }
        __syncthreads();
        if (hf == 0) {
            float add = 0.0f;
            for (int w = 0; w < (warp & 3); ++w) add += wsum[w];
            lg_s[r] += add;
        }
        __syncthreads();
        // ---- U_q, U_k, U_v of the tile (its copies went out while the tile before it was finished)
        if (tid == 0) {
            if (seg_first) ok = wait_bar(bars + 8 * kTRBarW, (segs - 1) & 1u, ab, 110);
            if (ok) ok = wait_bar(bars + 8 * kTRBarLoad, par, ab, 111);
            if (ok) {
                tc_fence_after();
#pragma unroll
                for (int u = 0; u < 3; ++u) {
                    const uint32_t a_lo = lo_of(kTROffQ + u * kTileBytes, kLboK), b_lo = lo_of(u * kTileBytes, kLboK);
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks)
                        mma_ss(tmem_base + u * kTile, desc64(a_lo + koff_k(ks)), desc64(b_lo + koff_k(ks)), idesc_kk, ks > 0);
                }
                mma_commit(bars + 8 * kTRBarU);
            }
        }
        const float lg_last = lg_s[kTile - 1];
        const float lg_r = lg_s[r];
        const float la_r = r > 0 ? lg_s[r - 1] : 0.0f;

        alive = wait_bar(bars + 8 * kTRBarU, par, ab, 112);
        if (alive) {
            tc_fence_after();
            // ---- pass 1: Q' and Khat (norm over the whole row, this thread keeps its half), V'
            uint32_t x[64];
#pragma unroll
            for (int t = 0; t < 2; ++t) {   // t = 0: Q, t = 1: K
                float ss4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
                for (int part = 0; part < 2; ++part) {
                    const int col = (part == 0 ? (hf ^ 1) : hf) * 64;
                    tmem_ld32(lane_base + t * kTile + col, *reinterpret_cast<uint32_t(*)[32]>(&x[0]));
                    tmem_ld32(lane_base + t * kTile + col + 32, *reinterpret_cast<uint32_t(*)[32]>(&x[32]));
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 64; i += 4) {
#pragma unroll
                        for (int e = 0; e < 4; ++e) ss4[e] = fmaf(__uint_as_float(x[i + e]), __uint_as_float(x[i + e]), ss4[e]);
                    }
                }
                float f = rsqrtf((ss4[0] + ss4[1]) + (ss4[2] + ss4[3]) + p.s.eps);
                if (t == 1) f *= __expf(lg_last - lg_r);          // Khat_j = w_j K'_j
                if (p.rope_h != nullptr) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const uint32_t h2[4] = {cs[i].x, cs[i].y, cs[i].z, cs[i].w};
#pragma unroll
                        for (int m = 0; m < 4; ++m) {
                            float cc, s1;
                            unpack_cs(h2[m], cc, s1);
                            const int at = i * 8 + 2 * m;
                            const float x0 = __uint_as_float(x[at]), x1 = __uint_as_float(x[at + 1]);
                            x[at] = __float_as_uint(x0 * cc - x1 * s1);
                            x[at + 1] = __float_as_uint(x0 * s1 + x1 * cc);
                        }
                    }
                }
                store_half_row_bf16_swizzled(smem + kTROffQ + t * kTileBytes, r, hf, x, f);
            }
            tmem_ld32(lane_base + kColV + hf * 64, *reinterpret_cast<uint32_t(*)[32]>(&x[0]));
            tmem_ld32(lane_base + kColV + hf * 64 + 32, *reinterpret_cast<uint32_t(*)[32]>(&x[32]));
            tmem_wait_ld();
            store_half_row_bf16_swizzled(smem + kTROffV, r, hf, x, 1.0f);
            // ---- Shat = exp(lg_last) S: back into TMEM (row d = r) and as a bf16 operand copy
            const float g_last = __expf(lg_last);
            tmem_ld32(lane_base + kColS + hf * 64, *reinterpret_cast<uint32_t(*)[32]>(&x[0]));
            tmem_ld32(lane_base + kColS + hf * 64 + 32, *reinterpret_cast<uint32_t(*)[32]>(&x[32]));
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 64; ++i) x[i] = __float_as_uint(__uint_as_float(x[i]) * g_last);
            tmem_st32(lane_base + kColS + hf * 64, *reinterpret_cast<uint32_t(*)[32]>(&x[0]));
            tmem_st32(lane_base + kColS + hf * 64 + 32, *reinterpret_cast<uint32_t(*)[32]>(&x[32]));
            store_half_row_bf16_swizzled(smem + kTROffS, r, hf, x, 1.0f);
            tmem_wait_st();
        }
        fence_proxy_async_smem();
        tc_fence_before();
        if (__syncthreads_or(!alive)) break;   // every thread leaves together
        // ---- SC = Q' Khat^T (columns of U_q), O = Q' Shat (columns of U_k)
        if (tid == 0 && ok) {
            tc_fence_after();
            const uint32_t q_lo = lo_of(kTROffQ, kLboK), k_lo = lo_of(kTROffK, kLboK), s_lo = lo_of(kTROffS, kLboMN);
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
                mma_ss(tmem_base + kColQ, desc64(q_lo + koff_k(ks)), desc64(k_lo + koff_k(ks)), idesc_kk, ks > 0);
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
                mma_ss(tmem_base + kColK, desc64(q_lo + koff_k(ks)), desc64(s_lo + koff_n(ks)), idesc_kn, ks > 0);
            mma_commit(bars + 8 * kTRBarA);
        }
        alive = wait_bar(bars + 8 * kTRBarA, par, ab, 113);
        if (tid == 0 && ok && alive) {
            // Shat's operand copy has been read: what the softmax branch left in these rows comes in its place, under pass 2 and the MMAs
            // after it, and the sums leave from there, both by TMA.  Row by row from the threads, 32 bytes at a time and
            // asked for ahead, the epilogue took 3.0 k of a tile's 13.5 k clk (by 16, when needed, 7.9 k of 17.7 k): 40 heads x 1500 tokens
            // 136.8 -> 131.4 us per pass, 8 x 12 x 700 116.2 -> 112.6, 12 x 1560 the same (one tile per CTA)
            const uint32_t bar = bars + 8 * kTRBarOut;
            mbar_expect_tx(bar, kTileBytes);
#pragma unroll
            for (int w = 0; w < 8; ++w)
                tma_load_4d(smem_base + kTROffS + (w >> 2) * kHalfBytes + (w & 3) * 32 * 128, &tm_o, bar, (w >> 2) * 64, h, tl * kTile + (w & 3) * 32, b);
            ++out_loads;
        }
        if (alive) {
            tc_fence_after();
            // ---- pass 2: P = strictly lower triangle of SC (keys hf * 64 ..), bf16 pairs into the U_v columns
            uint32_t sc[64], pk[32];
            tmem_ld32(lane_base + kColQ + hf * 64, *reinterpret_cast<uint32_t(*)[32]>(&sc[0]));
            tmem_ld32(lane_base + kColQ + hf * 64 + 32, *reinterpret_cast<uint32_t(*)[32]>(&sc[32]));
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                const int j0 = hf * 64 + 2 * i;
                pk[i] = pack_bf16(j0 < r ? __uint_as_float(sc[2 * i]) : 0.0f, j0 + 1 < r ? __uint_as_float(sc[2 * i + 1]) : 0.0f);
            }
            tmem_st32(lane_base + kColV + hf * 32, pk);
            tmem_wait_st();
        }
        tc_fence_before();
        if (__syncthreads_or(!alive)) break;
        // ---- O += P V',  S += Khat^T V'
        if (tid == 0 && ok) {
            tc_fence_after();
            const uint32_t v_lo = lo_of(kTROffV, kLboMN), k_lo = lo_of(kTROffK, kLboMN);
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
                mma_ts(tmem_base + kColK, tmem_base + kColV + ks * 8, desc64(v_lo + koff_n(ks)), idesc_kn, 1u);
            if (!seg_last) {
#pragma unroll
                for (int ks = 0; ks < 8; ++ks)
                    mma_ss(tmem_base + kColS, desc64(k_lo + koff_n(ks)), desc64(v_lo + koff_n(ks)), idesc_nn, 1u);
            }
            mma_commit(bars + 8 * kTRBarB);
        }
        alive = wait_bar(bars + 8 * kTRBarB, par, ab, 114);
        if (tid == 0 && ok && alive && g + 1 < g_end) {
            // every MMA that read the tiles is done: the next ones land under the epilogue
            load_tiles(g + 1);
            ++loads;
            if (tl + 1 == p.ntile) {
                load_maps((g + 1) / p.ntile % H);
                ++map_loads;
            }
        }
        const float sig = row < L ? sigmoid_fast(gate_logit) : 0.0f;
        if (g + 1 < g_end) fetch_row(g + 1);
        alive = alive && wait_bar(bars + 8 * kTRBarOut, par, ab, 115);
        if (__all_sync(0xffffffffu, alive)) {
            tc_fence_after();
            // ---- epilogue: out_i += sigmoid(g_i) exp(la_i - lg_last) O_i
            uint32_t o[64];
            tmem_ld32(lane_base + kColK + hf * 64, *reinterpret_cast<uint32_t(*)[32]>(&o[0]));
            tmem_ld32(lane_base + kColK + hf * 64 + 32, *reinterpret_cast<uint32_t(*)[32]>(&o[32]));
            tmem_wait_ld();
            const float f = sig * __expf(la_r - lg_last);
            uint8_t* half_row = smem + kTROffS + hf * kHalfBytes + r * 128;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                uint4* piece = reinterpret_cast<uint4*>(half_row + ((i ^ (r & 7)) << 4));
                const uint4 v = *piece;
                const uint32_t prev[4] = {v.x, v.y, v.z, v.w};
                uint32_t nw[4];
#pragma unroll
                for (int m = 0; m < 4; ++m)
                    nw[m] = pack_bf16(__uint_as_float(prev[m] << 16) + f * __uint_as_float(o[i * 8 + 2 * m]),
                                      __uint_as_float(prev[m] & 0xFFFF0000u) + f * __uint_as_float(o[i * 8 + 2 * m + 1]));
                *piece = make_uint4(nw[0], nw[1], nw[2], nw[3]);
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0 && row < L)   // this warp's 32 rows; those past the end stay away
                tma_store_4d(&tm_o, smem_base + kTROffS + hf * kHalfBytes + r * 128, hf * 64, h, row, b);
        }
        tc_fence_before();
        if (__syncthreads_or(!alive)) break;   // the tiles and the gate arrays may be overwritten now
    }
    if (lane == 0) tma_store_wait_read();
    if (tid == 0 && (!ok || *abort_flag)) {
        // leave no bulk copy in flight into this CTA's shared memory, no MMA writing tensor memory
        drain_bar(bars + 8 * kTRBarW, (uint32_t)(map_loads - 1) & 1u);
        if (loads > 0) drain_bar(bars + 8 * kTRBarLoad, (uint32_t)(loads - 1) & 1u);
        if (out_loads > 0) drain_bar(bars + 8 * kTRBarOut, (uint32_t)(out_loads - 1) & 1u);
        mma_commit(bars + 8 * kTRBarDrain);
        drain_bar(bars + 8 * kTRBarDrain, 0);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

std::mutex g_setup_mutex;
DeviceSetup g_setup[kMaxDevices];

}  // namespace

int tc_token_readout(const StepArgs& a, const float* alpha_logits, const CommitArgs& seg, const __nv_bfloat16* wq_op,
                     const __nv_bfloat16* wk_op, const __nv_bfloat16* wv_op, cudaStream_t st)
{
    int num_sms = 0;
    if (int r = device_setup_once(g_setup_mutex, g_setup,
                                  [] { return opt_in_smem(tc_token_readout_kernel, kTRSmemBytes); }, &num_sms))
        return r;
    CUtensorMap tm_q, tm_k, tm_v, tm_wq, tm_wk, tm_wv, tm_o;
    if (int r = make_map_blhd(&tm_q, a.q, a.s)) return r;
    if (int r = make_map_blhd(&tm_k, a.k_rot, a.s)) return r;     // raw K: the feature map comes before the rotation
    if (int r = make_map_blhd(&tm_v, a.v, a.s)) return r;
    if (int r = make_map_blhd(&tm_o, a.out, a.s, 32)) return r;
    if (int r = make_map_rows(&tm_wq, wq_op, (size_t)a.s.H * kTile)) return r;
    if (int r = make_map_rows(&tm_wk, wk_op, (size_t)a.s.H * kTile)) return r;
    if (int r = make_map_rows(&tm_wv, wv_op, (size_t)a.s.H * kTile)) return r;
    TcReadoutParams p;
    p.s = a.s;
    p.rope_h = static_cast<const uint4*>(a.rope_h);
    p.alpha = alpha_logits;
    p.gate = a.gate;
    p.state = a.state;
    p.entry = seg.partials;
    p.status = a.status;
    p.spin_limit = a.wait_limit ? a.wait_limit - 1 : kSpinLimit;
    p.ntile = seg.run_ntile;
    p.share = seg.run_share;
    p.nslot = seg.nslot;
    p.total_tiles = a.s.B * a.s.H * p.ntile;
    const int grid = (p.total_tiles + p.share - 1) / p.share;
    const cudaError_t e = launch_kernel(tc_token_readout_kernel, dim3((unsigned)grid), kTRThreads, kTRSmemBytes, st, tm_q, tm_k, tm_v, tm_wq,
                                        tm_wk, tm_wv, tm_o, p);
    if (e != cudaSuccess) { set_error("launch of tc_token_readout_kernel failed: %s", cudaGetErrorString(e)); return ARL2_ERR_CUDA; }
    return 1;
}

}  // namespace arl2
