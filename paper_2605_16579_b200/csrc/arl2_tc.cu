// Tensor-core (tcgen05 / TMEM / TMA) kernels of the ARL^2 layer for bf16 I/O, D = 128.
//
// Step kernel (Eq. 2, 3, 5-8): persistent, one CTA per SM.  A work item drives two 128-row query
// tiles: two consecutive tiles of one (stream, head), or the ragged last tiles of two different
// (stream, head) units.  Items are handed out by an atomic counter, the pairs first.
//   warps 0-3 / 4-7  softmax group of query tile 0 / 1 (one thread per query row)
//   warp 8           TMA producer and scheduler: the Q tiles, then through a 5-slot ring K_j, V_j
//                    for every key tile, then W_phi_q^T, the raw Q tiles again and the bf16
//                    copy of the state S
//   warp 9 / 10      MMA issuer of tile 0 / 1 (the warp walks the loop, one elected lane issues):
//                    S_t = Q~_t K_j^T and O_t += P_t V_j into TMEM
// TMEM (512 columns): S_0 | S_1 | O_0 | O_1, 128 fp32 columns each; the bf16 probabilities P_t
// overwrite the first 64 columns of S_t and feed the second MMA straight from TMEM.
// RoPE(Q) is applied in place in shared memory by the softmax groups; K arrives rotated.
// The inter branch reuses the loop as one more iteration: "S" = Q W_phi_q (A = the raw Q tile
// from the ring), the group turns each row into sigmoid(g) * l * L2Norm(RoPE(.)) (l = softmax
// row sum) and the "PV" MMA multiplies it by the state, accumulating into O_t, so that the
// final O_t / l is O_intra + sigmoid(g) O_inter.  The state is only read.
//
// Every wait is bounded: when a limit expires the thread records ARL2_ERR_TIMEOUT in the
// device status block, raises the CTA's abort flag and every role falls through to the exit.
#include <type_traits>

#include "tc_common.cuh"

namespace arl2 {

namespace {

constexpr int kStages = 5;
constexpr int kThreads = 384;              // 3 warpgroups: softmax 0, softmax 1, {TMA, MMA, 2 idle}
constexpr int kRegsSoftmax = 232;          // per-thread registers after the warpgroups rebalance
constexpr int kRegsOther = 40;
// setmaxnreg.inc waits (without a bound) for registers of the CTA's own launch allocation
// (threads x the launch register count): the rebalanced total must fit in it
constexpr int kLaunchRegs = (65536 / kThreads) / 8 * 8;
static_assert(256 * kRegsSoftmax + (kThreads - 256) * kRegsOther <= kThreads * kLaunchRegs, "register pool");
constexpr float kRescaleThreshold = 8.0f;   // log2 units of slack before O is rescaled

// shared memory map (offsets from a 1024-byte aligned base)
constexpr int kOffQ = 0;                                 // 2 query tiles (rotated in place)
constexpr int kOffRing = kOffQ + 2 * kTileBytes;         // kStages tiles
constexpr int kOffBars = kOffRing + kStages * kTileBytes;
constexpr int kSmemBytes = kOffBars + 256 + 1024;        // barriers + alignment slack

enum Bar : int {
    kBarQFull = 0,                              // producer -> all: Q tiles (and the item id) landed
    kBarQFree,                                  // MMA -> producer: last MMA reading Q~ is done
    kBarQRot0, kBarQRot1,                       // softmax group t -> MMA: Q~_t rotated
    kBarFull0,                                  // kStages of them
    kBarEmpty0 = kBarFull0 + kStages,           // kStages of them
    kBarSFull0 = kBarEmpty0 + kStages, kBarSFull1,
    kBarPFull0, kBarPFull1,
    kBarOFinal0, kBarOFinal1,
    kBarTurn0, kBarTurn1,                       // the MMA issuers take turns on the tensor pipe
    kBarDrain0, kBarDrain1,                     // an MMA issuer that gives up waits here for its MMAs in flight
    kNumBars
};
// after the barriers: TMEM base (4 B), abort flag (4 B), two item-id slots (8 B)
static_assert(kNumBars * 8 + 16 <= 256, "barrier block");

struct TcStepParams {
    Shape s;
    const float* gate;
    const float* rope_cos;
    const float* rope_sin;
    const uint4* rope_h;       // half2 (cos, sin) table, warp-interleaved (see pack_rope_kernel), or nullptr
    __nv_bfloat16* out;
    uint32_t* status;
    uint32_t spin_limit;       // polls a bounded wait makes before it gives up
    int k_made_before;         // the kernel before this one made K and nothing else that is read or written here
    uint32_t* sched_counter;   // this launch's item counter (zero on entry, and again once every item has run)
    uint32_t* sched_next;      // the next launch's counter: cleared by this launch (the one before may have given up on a wait)
    int gate_mode;             // 0: gate logits [B, L, H]; 1: [B, L] (one per token); 2: [B, L, H, D] (per channel)
    int Lk;                    // keys per head: L, or the length of a key/value cache (Eq. 1)
    int n_q;                   // query tiles per head
    int n_kv;                  // key tiles per head
    int n_pair_items;          // B * H * (n_q / 2): items with two query tiles
    int n_items;               // + ceil(B * H / 2) items of ragged last tiles when n_q is odd
    // Key-range split of the last wave: items [0, n_whole) run whole; item n_whole + s (s = "slot")
    // runs as k_split parts over consecutive ranges of key tiles, scheduled as ids n_whole +
    // s * k_split + part.  Every part leaves its unnormalised rows, reference maxima and row sums in
    // the split buffers; tc_split_merge_kernel then combines the parts of a row in index order.
    int n_whole;
    int k_split;               // 1: nothing is split
    int one_item;              // every CTA has one item: the query tiles' shared memory is free for its output
    int n_sched;               // ids the scheduler hands out: n_whole + (n_items - n_whole) * k_split
    float* split_o;            // [slot][tile][part][128 rows][128] unnormalised output rows
    float* split_ml;           // [slot][tile][part][128 rows][2] reference maximum (log2 units), row sum
};

// A work item drives up to two 128-row query tiles.  A "pair" item holds two consecutive tiles of
// one (stream, head): they share every K/V tile.  A "ragged" item holds the last, partial tiles
// of two different (stream, head) units (or of one, when the number of units is odd): each tile
// then streams its own K/V, W_phi_q and state through the ring.
struct Item {
    int b[2], h[2], row0[2];
    int ntile;    // active tiles: 1 or 2
    bool shared;  // both tiles read the same K, V, W_phi_q and state
    int j0, nj;   // key tiles [j0, j0 + nj) of the head
    int part;     // -1: the whole key range; else index of this part
    int slot;     // split items only: index among the split items
};

// Items [0, n_pair_items) are pairs of full tiles, (b, h)-major so that neighbours share K and V
// in L2; the rest pack the ragged last tiles two by two.
template <bool kSplit>
__device__ __forceinline__ Item decode_item(int id, const TcStepParams& p)
{
    Item it;
    it.j0 = 0;
    it.nj = p.n_kv;
    it.part = -1;
    it.slot = 0;
    if (kSplit && id >= p.n_whole) {
        const int x = id - p.n_whole;
        it.slot = x / p.k_split;
        it.part = x - it.slot * p.k_split;
        id = p.n_whole + it.slot;
        it.j0 = (it.part * p.n_kv) / p.k_split;
        it.nj = ((it.part + 1) * p.n_kv) / p.k_split - it.j0;
    }
    const int full_pairs = p.n_q >> 1;
    const int units = p.s.B * p.s.H;
    if (id < p.n_pair_items) {
        const int bh = id / full_pairs;
        const int pair = id - bh * full_pairs;
        it.b[0] = it.b[1] = bh / p.s.H;
        it.h[0] = it.h[1] = bh - it.b[0] * p.s.H;
        it.row0[0] = pair * 2 * kTile;
        it.row0[1] = it.row0[0] + kTile;
        it.ntile = 2;
        it.shared = true;
    } else {
        const int u = id - p.n_pair_items;
        it.ntile = (2 * u + 1 < units) ? 2 : 1;
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const int bh = min(2 * u + t, units - 1);
            it.b[t] = bh / p.s.H;
            it.h[t] = bh - it.b[t] * p.s.H;
            it.row0[t] = full_pairs * 2 * kTile;
        }
        it.shared = false;
    }
    return it;
}

// The ring entries of an item, in the order both MMA issuers walk them.
enum EntryKind : int { kEntK = 0, kEntV, kEntW, kEntQRaw, kEntState };
struct Entry {
    int kind, tile, j;   // j: key tile index for K / V
};
// pair item:   K_0 | V_0 K_1 | V_1 K_2 | ... | V_{n-1} W Qraw_0 Qraw_1 | S
// ragged item: K^0_0 K^1_0 | V^0_0 K^0_1 V^1_0 K^1_1 | ... | V^0_{n-1} W^0 Qraw_0 V^1_{n-1} W^1 Qraw_1 | S^0 S^1
__device__ __forceinline__ int item_entries(const Item& it, int n_kv)
{
    return it.shared ? 2 * n_kv + 2 + it.ntile : it.ntile * (2 * n_kv + 3);
}
__device__ __forceinline__ Entry item_entry(const Item& it, int n_kv, int e)
{
    Entry en;
    if (it.shared) {
        en.tile = 0;
        if (e == 0) { en.kind = kEntK; en.j = 0; }
        else if (e < 2 * n_kv) { en.kind = (e & 1) ? kEntV : kEntK; en.j = (e & 1) ? (e - 1) >> 1 : e >> 1; }
        else if (e == 2 * n_kv) { en.kind = kEntW; en.j = 0; }
        else if (e < 2 * n_kv + 1 + it.ntile) { en.kind = kEntQRaw; en.tile = e - (2 * n_kv + 1); en.j = 0; }
        else { en.kind = kEntState; en.j = 0; }
    } else {
        const int nt = it.ntile;
        const int body = nt + 2 * nt * (n_kv - 1);   // entries before the last key iteration
        if (e < nt) { en.kind = kEntK; en.tile = e; en.j = 0; }
        else if (e < body) {
            const int x = e - nt, jj = x / (2 * nt), y = x - jj * 2 * nt;
            en.tile = y >> 1;
            en.kind = (y & 1) ? kEntK : kEntV;
            en.j = (y & 1) ? jj + 1 : jj;
        } else if (e < body + 3 * nt) {
            const int y = e - body;
            en.tile = y / 3;
            const int z = y - en.tile * 3;
            en.kind = z == 0 ? kEntV : z == 1 ? kEntW : kEntQRaw;
            en.j = n_kv - 1;
        } else { en.kind = kEntState; en.tile = e - (body + 3 * nt); en.j = 0; }
    }
    return en;
}

// One softmax group thread: owns query row `r` of tile `t` of every item.  kElemGate: one gate
// per output channel, which only launches with such gates take (a kernel instantiation of its own, with that epilogue alone).
// No lane leaves it alone when a wait expires: the lanes meet again (the vote on rescaling, the box of output rows that leaves by
// TMA), and the others would wait for it for good.  In the key loop the role goes on instead; the error is recorded, the waits
// after it end at once, and the next one behind the loop ends the role for the whole warp.  Lanes that left by themselves,
// a whole-warp wait in the loop too, and this: 40 heads x 4680 tokens 454, 461, 457 us, 8 x 12 x 4680 1071, 1084, 1076, attention over a
// cache of 4 x 4680 tokens 498, 499, 502; shorter ones the same.
template <bool kElemGate, bool kSplit>
__device__ __forceinline__ void softmax_role(const TcStepParams& p, const CUtensorMap* tm_o, uint8_t* smem, uint32_t bars,
                                             uint32_t tmem_base, const Abort& ab,
                                             const volatile int* item_slots, int t, int r,
                                             int warp_in_group)
{
    const int L = p.s.L, H = p.s.H;
    const uint32_t lane_base = tmem_base + ((uint32_t)(warp_in_group * 32) << 16);
    const uint32_t s_addr = lane_base + (uint32_t)(t * kTile);
    const uint32_t o_addr = lane_base + (uint32_t)(2 * kTile + t * kTile);
    const uint32_t bar_s = bars + 8 * (kBarSFull0 + t);
    const uint32_t bar_p = bars + 8 * (kBarPFull0 + t);
    const float c2 = p.s.scale_log2;
    const uint64_t c2x2 = pack2(c2, c2);
    const int n_kv = p.n_kv;
    uint32_t s_cnt = 0;   // phases of bar_s consumed so far
    uint32_t of_cnt = 0;  // phases of this tile's final-O barrier consumed so far
    uint32_t sreg[128];

    for (uint32_t item = 0;; ++item) {
        // the first item is known without the producer: its rotation table is fetched while Q is on its way (a rotation
        // that asked for the table once Q had landed ended 1.2 us later)
        if (item > 0 && !wait_bar_warp(bars + 8 * kBarQFull, item & 1, ab, 10)) return;
        const int id = item > 0 ? item_slots[item & 1] : (int)blockIdx.x;
        if (id < 0) return;
        const Item it = decode_item<kSplit>(id, p);
        const int j0 = kSplit ? it.j0 : 0, nj = kSplit ? it.nj : n_kv;
        const int b = it.b[t], h = it.h[t];
        const int row = it.row0[t] + r;
        const bool valid_row = row < L;
        const bool active = t < it.ntile;
        if (item == 0 && !active && !wait_bar_warp(bars + 8 * kBarQFull, 0, ab, 10)) return;   // (no phase is left out)

        if (active) {
            // ---- Q~ = RoPE(Q): rotate this thread's row of the tile in place          (Eq. 2)
            if (p.rope_h != nullptr) {
                uint8_t* tile = smem + kOffQ + t * kTileBytes;
                // all 16 table loads of the row go out before the first one is used
                const uint4* tab = p.rope_h + ((size_t)(row >> 5) * 16) * 32 + (row & 31);
                uint4 cs[16];
#pragma unroll
                for (int c = 0; c < 16; ++c) cs[c] = tab[c * 32];
                if (item == 0 && !wait_bar_warp(bars + 8 * kBarQFull, 0, ab, 10)) return;
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    int off = (c >> 3) * kHalfBytes + r * 128 + (((c & 7) ^ (r & 7)) << 4);
                    uint4 raw = *reinterpret_cast<const uint4*>(tile + off);
                    uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
                    const uint32_t h2[4] = {cs[c].x, cs[c].y, cs[c].z, cs[c].w};
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        float cc, ss;
                        unpack_cs(h2[m], cc, ss);
                        float x0 = __uint_as_float(w[m] << 16);
                        float x1 = __uint_as_float(w[m] & 0xFFFF0000u);
                        w[m] = pack_bf16(x0 * cc - x1 * ss, x0 * ss + x1 * cc);
                    }
                    *reinterpret_cast<uint4*>(tile + off) = make_uint4(w[0], w[1], w[2], w[3]);
                }
                fence_proxy_async_smem();
            } else if (item == 0 && !wait_bar_warp(bars + 8 * kBarQFull, 0, ab, 10)) {
                return;
            }
            mbar_arrive(bars + 8 * (kBarQRot0 + t));

            float m_ref = -INFINITY;   // reference maximum (scaled, base 2) of the probabilities
            uint64_t l2 = pack2(0.0f, 0.0f);   // running row sum relative to m_ref, two lanes

            for (int jj = 0; jj < nj; ++jj) {
                const int j = j0 + jj;
                (void)wait_bar(bar_s, s_cnt & 1, ab, 20 + t);   // (where it expired, the loop goes on over whatever is there)
                ++s_cnt;
                tc_fence_after();
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    tmem_ld32(s_addr + c * 32, *reinterpret_cast<uint32_t(*)[32]>(&sreg[c * 32]));
                tmem_wait_ld();

                const int n_valid = p.Lk - j * kTile;  // keys of this tile that exist
                if (n_valid < kTile) {   // ragged last tile: zero-filled key rows must not count
#pragma unroll
                    for (int c = 0; c < 128; ++c)
                        if (c >= n_valid) sreg[c] = __float_as_uint(-INFINITY);
                }
                float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
                for (int c = 0; c < 128; c += 8) {
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        m4[k] = max3(m4[k], __uint_as_float(sreg[c + 2 * k]), __uint_as_float(sreg[c + 2 * k + 1]));
                }
                const float mx = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
                const float m_new = fmaxf(m_ref, mx * c2);
                const bool need = (m_new - m_ref) > kRescaleThreshold;   // first tile: inf > threshold
                if (__any_sync(0xffffffffu, need)) {
                    float alpha = 1.0f;
                    if (need) {
                        alpha = ex2_approx(m_ref - m_new);
                        m_ref = m_new;
                        l2 = fma2(l2, pack2(alpha, alpha), pack2(0.0f, 0.0f));
                    }
                    if (jj > 0) {
                        // the MMA that last accumulated into O_t finished before S_t(j) was
                        // signalled, and the next one waits for this group's arrival below
#pragma unroll 1
                        for (int c = 0; c < 4; ++c) {
                            uint32_t o[32];
                            tmem_ld32(o_addr + c * 32, o);
                            tmem_wait_ld();
#pragma unroll
                            for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
                            tmem_st32(o_addr + c * 32, o);
                        }
                    }
                }
                const uint64_t neg_m2 = pack2(-m_ref, -m_ref);
#pragma unroll
                for (int c = 0; c < 64; ++c) {
                    float x0, x1, p0, p1;
                    unpack2(fma2(pack2(__uint_as_float(sreg[2 * c]), __uint_as_float(sreg[2 * c + 1])), c2x2, neg_m2),
                            x0, x1);
                    p0 = ex2_approx(x0);
                    p1 = ex2_approx(x1);
                    l2 = add2(l2, pack2(p0, p1));
                    sreg[c] = pack_bf16(p0, p1);
                }
                tmem_st32(s_addr, *reinterpret_cast<uint32_t(*)[32]>(&sreg[0]));
                tmem_st32(s_addr + 32, *reinterpret_cast<uint32_t(*)[32]>(&sreg[32]));
                tmem_wait_st();
                tc_fence_before();
                mbar_arrive(bar_p);
            }
            float l_lo, l_hi;
            unpack2(l2, l_lo, l_hi);
            const float l_sum = l_lo + l_hi;

            // ---- inter branch: U = Q W_phi_q arrives in the S columns                  (Eq. 3)
            // the row's rotation table is fetched while the MMA is still running
            uint4 cs[16];
            // fetched early too; no gate tensor = closed gate (plain softmax attention, Eq. 1)
            const float gate_logit = (valid_row && p.gate != nullptr && !kElemGate)
                                         ? p.gate[p.gate_mode == 1 ? (size_t)b * L + row : ((size_t)b * L + row) * H + h]
                                         : -INFINITY;
            const bool rotate_u = p.rope_h != nullptr && valid_row;
            if (rotate_u) {
                const uint4* tab = p.rope_h + ((size_t)(row >> 5) * 16) * 32 + (row & 31);
#pragma unroll
                for (int c = 0; c < 16; ++c) cs[c] = tab[c * 32];
            }
            if (!wait_bar_warp(bar_s, s_cnt & 1, ab, 30 + t)) return;
            ++s_cnt;
            tc_fence_after();
#pragma unroll
            for (int c = 0; c < 4; ++c)
                tmem_ld32(s_addr + c * 32, *reinterpret_cast<uint32_t(*)[32]>(&sreg[c * 32]));
            tmem_wait_ld();
            {
                if (rotate_u) {
#pragma unroll
                    for (int c = 0; c < 16; ++c) {
                        const uint32_t h2[4] = {cs[c].x, cs[c].y, cs[c].z, cs[c].w};
#pragma unroll
                        for (int m = 0; m < 4; ++m) {
                            float cc, s1;
                            unpack_cs(h2[m], cc, s1);
                            float x0 = __uint_as_float(sreg[c * 8 + 2 * m]);
                            float x1 = __uint_as_float(sreg[c * 8 + 2 * m + 1]);
                            sreg[c * 8 + 2 * m] = __float_as_uint(x0 * cc - x1 * s1);
                            sreg[c * 8 + 2 * m + 1] = __float_as_uint(x0 * s1 + x1 * cc);
                        }
                    }
                }
                float ss4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
                for (int c = 0; c < 128; c += 4) {
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        ss4[k] = fmaf(__uint_as_float(sreg[c + k]), __uint_as_float(sreg[c + k]), ss4[k]);
                }
                const float ss = (ss4[0] + ss4[1]) + (ss4[2] + ss4[3]);
                const float gate = valid_row ? sigmoid_fast(gate_logit) : 0.0f;
                // scaled by the row sum so that the common 1/l of the epilogue leaves gate * Q' S;
                // with per-channel gates the readout is kept apart and gated in the epilogue
                const float f = kElemGate ? rsqrtf(ss + p.s.eps) : rsqrtf(ss + p.s.eps) * gate * l_sum;
#pragma unroll
                for (int c = 0; c < 64; ++c)
                    sreg[c] = pack_bf16(__uint_as_float(sreg[2 * c]) * f, __uint_as_float(sreg[2 * c + 1]) * f);
            }
            tmem_st32(s_addr, *reinterpret_cast<uint32_t(*)[32]>(&sreg[0]));
            tmem_st32(s_addr + 32, *reinterpret_cast<uint32_t(*)[32]>(&sreg[32]));
            tmem_wait_st();
            tc_fence_before();
            mbar_arrive(bar_p);

            if constexpr (kElemGate) {
                // ---- per-channel gates: X = Q' S arrives 64 channels at a time in columns 64-127 of
                // S_t; out = O_t / l + sigmoid(G) X.  O_t is final: its last MMA preceded U's.
                const float inv_l = 1.0f / l_sum;
                const size_t rbase = ((size_t)b * L + (valid_row ? row : 0)) * H + h;
                __nv_bfloat16* orow = p.out + rbase * kTile;
                const float* grow = p.gate + rbase * kTile;
                // The logits may start at any element and the output rows on any 16 bytes: decided once per 32 channels.  At each
                // access, 40 heads x 1560 tokens took 114.1 us against 113.4 without the choice; so, and without the other
                // epilogues in this instantiation, 112.2 (12 x 1560: 55.6, 55.0 and 54.6).
                const bool wide = (reinterpret_cast<uintptr_t>(p.gate) & 15) == 0 && wide_rows(p.out);
#pragma unroll 1
                for (int hv = 0; hv < 2; ++hv) {
                    if (!wait_bar_warp(bar_s, s_cnt & 1, ab, 32 + t)) return;
                    ++s_cnt;
                    tc_fence_after();
#pragma unroll 1
                    for (int c = 0; c < 2; ++c) {
                        uint32_t x[32], o[32];
                        tmem_ld32(s_addr + 64 + c * 32, x);
                        tmem_ld32(o_addr + hv * 64 + c * 32, o);
                        tmem_wait_ld();
                        const int at = hv * 64 + c * 32;
                        if (valid_row && wide) {
#pragma unroll
                            for (int e = 0; e < 2; ++e) {
                                uint32_t w[8];
#pragma unroll
                                for (int i = 0; i < 4; ++i) {
                                    const float4 gl = *reinterpret_cast<const float4*>(grow + at + e * 16 + i * 4);
                                    const float gv[4] = {gl.x, gl.y, gl.z, gl.w};
                                    float y[4];
#pragma unroll
                                    for (int u = 0; u < 4; ++u) {
                                        const int n = e * 16 + i * 4 + u;
                                        y[u] = __uint_as_float(o[n]) * inv_l + sigmoid_fast(gv[u]) * __uint_as_float(x[n]);
                                    }
                                    w[i * 2] = pack_bf16(y[0], y[1]);
                                    w[i * 2 + 1] = pack_bf16(y[2], y[3]);
                                }
                                store_row32(orow + at + e * 16, w);
                            }
                        } else if (valid_row) {
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                uint32_t w[4];
#pragma unroll
                                for (int i = 0; i < 4; ++i) {
                                    const int n = e * 8 + i * 2;
                                    const float* gp = grow + at + n;
                                    w[i] = pack_bf16(__uint_as_float(o[n]) * inv_l + sigmoid_fast(gp[0]) * __uint_as_float(x[n]),
                                                     __uint_as_float(o[n + 1]) * inv_l + sigmoid_fast(gp[1]) * __uint_as_float(x[n + 1]));
                                }
                                *reinterpret_cast<uint4*>(orow + at + e * 8) = make_uint4(w[0], w[1], w[2], w[3]);
                            }
                        }
                    }
                    tc_fence_before();
                    if (hv == 0) mbar_arrive(bar_p);   // the first half of X has been read
                }
                continue;
            }
            // ---- epilogue: O_t / l -> bf16 -> global                              (Eq. 6-7)
            if (!wait_bar_warp(bars + 8 * (kBarOFinal0 + t), of_cnt & 1, ab, 40 + t)) return;
            ++of_cnt;
            tc_fence_after();
            __nv_bfloat16* orow = p.out + (((size_t)b * L + (valid_row ? row : 0)) * H + h) * kTile;
            if (kSplit && it.part >= 0) {
                // ---- one part of a split item: its rows of O_t, unnormalised (the readout in them
                // is scaled by this part's row sum, so that the merged sum carries gate * Q' S times
                // the total row sum), the reference maximum and the row sum go to the split buffers;
                // tc_split_merge_kernel combines the parts
                const size_t tp = ((size_t)it.slot * 2 + t) * p.k_split + it.part;
                float* mine = p.split_o + (tp * kTile + r) * kTile;
#pragma unroll 1
                for (int c = 0; c < 4; ++c) {
                    uint32_t o[32];
                    tmem_ld32(o_addr + c * 32, o);
                    tmem_wait_ld();
                    if (valid_row) {
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(
                                             mine + c * 32 + e * 8),
                                         "r"(o[e * 8]), "r"(o[e * 8 + 1]), "r"(o[e * 8 + 2]), "r"(o[e * 8 + 3]),
                                         "r"(o[e * 8 + 4]), "r"(o[e * 8 + 5]), "r"(o[e * 8 + 6]), "r"(o[e * 8 + 7])
                                         : "memory");
                    }
                }
                tc_fence_before();
                if (valid_row) *reinterpret_cast<float2*>(p.split_ml + (tp * kTile + r) * 2) = make_float2(m_ref, l_sum);
                continue;
            }
            const float inv_l = 1.0f / l_sum;
            if (p.one_item && it.row0[t] + 96 < L) {
                // A row per thread makes a warp's stores 32 bytes of 32 rows each, which the load/store unit takes one by one: 3.8 k
                // clk for the two tiles, now 2.5 k.  Where no further item's Q is on its way, the rows go over this tile's Q
                // (every score MMA is done) and leave by TMA, 32 rows per warp; rows past L are cut off by the tensor map.
                // us per pass with row stores and so: 12 heads x 1560 tokens 38.7 and 38.3, 3 x 12 x 1001 32.6 and 32.4, 12 x 512 18.3
                // and 17.9, 2 x 384 17.7 and 17.5.  Only tiles in which all four warps have rows: the TMA's own latency is
                // there for a few rows, too, whose stores would be through sooner (12 x 300, 44 rows in the last tile,
                // 16.9 and 17.3; 12 x 330, 74 rows, 17.3 and 17.5).
                uint8_t* tile = smem + kOffQ + t * kTileBytes;
#pragma unroll 1
                for (int c = 0; c < 4; ++c) {
                    uint32_t o[32];
                    tmem_ld32(o_addr + c * 32, o);
                    tmem_wait_ld();
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        uint32_t w[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            w[i] = pack_bf16(__uint_as_float(o[q * 8 + 2 * i]) * inv_l, __uint_as_float(o[q * 8 + 2 * i + 1]) * inv_l);
                        const int v = (c & 1) * 4 + q;   // 16-byte piece of the 64-column box
                        *reinterpret_cast<uint4*>(tile + (c >> 1) * kHalfBytes + r * 128 + ((v ^ (r & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
                    }
                    if (c & 1) {   // the box is complete
                        fence_proxy_async_smem();
                        __syncwarp();
                        if ((r & 31) == 0 && row < L)
                            tma_store_4d(tm_o, smem_u32(tile) + (c >> 1) * kHalfBytes + r * 128, (c >> 1) * 64, h, row, b);
                    }
                }
                tc_fence_before();
                if ((r & 31) == 0) tma_store_wait_read();   // (the CTA ends soon)
                continue;
            }
            if (!wide_rows(p.out)) {
                // a loop of its own: with the choice at each store, attention over a cache of 4 x 4680 tokens took 512.4 us against
                // 509 without it (12 heads, 4680 queries); with this loop no difference is left
#pragma unroll 1
                for (int c = 0; c < 4; ++c) {
                    uint32_t o[32];
                    tmem_ld32(o_addr + c * 32, o);
                    tmem_wait_ld();
                    if (valid_row) {
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            uint32_t w[4];
#pragma unroll
                            for (int i = 0; i < 4; ++i)
                                w[i] = pack_bf16(__uint_as_float(o[e * 8 + 2 * i]) * inv_l, __uint_as_float(o[e * 8 + 2 * i + 1]) * inv_l);
                            *reinterpret_cast<uint4*>(orow + c * 32 + e * 8) = make_uint4(w[0], w[1], w[2], w[3]);
                        }
                    }
                }
                tc_fence_before();
                continue;
            }
#pragma unroll 1
            for (int c = 0; c < 4; ++c) {
                uint32_t o[32];
                tmem_ld32(o_addr + c * 32, o);
                tmem_wait_ld();
                if (valid_row) {
                    // 32-byte stores: each one fills a whole sector of the row
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        uint32_t w[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            w[i] = pack_bf16(__uint_as_float(o[e * 16 + 2 * i]) * inv_l,
                                             __uint_as_float(o[e * 16 + 2 * i + 1]) * inv_l);
                        store_row32(orow + c * 32 + e * 16, w);
                    }
                }
            }
            tc_fence_before();
        }
    }
}

template <bool kElemGate, bool kSplit>
__global__ void __launch_bounds__(kThreads, 1)
tc_step_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
               const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_w,
               const __grid_constant__ CUtensorMap tm_s, const __grid_constant__ CUtensorMap tm_o, const TcStepParams p)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                               ~static_cast<uintptr_t>(1023));
    const uint32_t smem_base = smem_u32(smem);
    const uint32_t bars = smem_base + kOffBars;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + kOffBars + kNumBars * 8);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + kOffBars + kNumBars * 8 + 4);
    volatile int* item_slots = reinterpret_cast<volatile int*>(smem + kOffBars + kNumBars * 8 + 8);
    const Abort ab{abort_flag, p.status, p.spin_limit};

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_kv = p.n_kv;

    if (!p.k_made_before) grid_dependency_sync();
    // a work item's Q tiles (and its id) for everyone who waits on kBarQFull
    auto request_q = [&](uint32_t slot, int id, const Item& it) {
        item_slots[slot] = id;
        const uint32_t bar_q = bars + 8 * kBarQFull;
        mbar_expect_tx(bar_q, it.ntile * kTileBytes);
        for (int t = 0; t < it.ntile; ++t) {
            const uint32_t dst = smem_base + kOffQ + t * kTileBytes;
            tma_load_4d(dst, &tm_q, bar_q, 0, it.h[t], it.row0[t], it.b[t]);
            tma_load_4d(dst + kHalfBytes, &tm_q, bar_q, 64, it.h[t], it.row0[t], it.b[t]);
        }
    };
    if (threadIdx.x == 8 * 32) {   // the TMA producer
        prefetch_tensormap(&tm_q);
        mbar_init(bars + 8 * kBarQFull, 1);
        mbar_init(bars + 8 * kBarQFree, 2);
        mbar_init(bars + 8 * kBarQRot0, 128);
        mbar_init(bars + 8 * kBarQRot1, 128);
        for (int s = 0; s < kStages; ++s) {
            mbar_init(bars + 8 * (kBarFull0 + s), 1);
            mbar_init(bars + 8 * (kBarEmpty0 + s), 2);   // both MMA issuers release every entry
        }
        mbar_init(bars + 8 * kBarSFull0, 1);
        mbar_init(bars + 8 * kBarSFull1, 1);
        mbar_init(bars + 8 * kBarPFull0, 128);
        mbar_init(bars + 8 * kBarPFull1, 128);
        mbar_init(bars + 8 * kBarOFinal0, 1);
        mbar_init(bars + 8 * kBarOFinal1, 1);
        mbar_init(bars + 8 * kBarTurn0, 1);
        mbar_init(bars + 8 * kBarTurn1, 1);
        mbar_init(bars + 8 * kBarDrain0, 1);
        mbar_init(bars + 8 * kBarDrain1, 1);
        *abort_flag = 0;
        fence_barrier_init();
        fence_proxy_async_smem();
        // the first item's Q goes out now, beside the allocation of tensor memory
        request_q(0, (int)blockIdx.x, decode_item<kSplit>((int)blockIdx.x, p));
        prefetch_tensormap(&tm_k);
        prefetch_tensormap(&tm_v);
        if (blockIdx.x == 0) *p.sched_next = 0;   // the next launch starts from a clean counter
    }
    if (warp == 9) {
        tmem_alloc(smem_u32(tmem_slot), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp < 8) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsSoftmax));
        softmax_role<kElemGate, kSplit>(p, &tm_o, smem, bars, tmem_base, ab, item_slots, warp >> 2, (warp & 3) * 32 + lane, warp & 3);
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsOther));
    }
    if (warp == 8) {
        // ---------------- TMA producer and scheduler ----------------
        if (lane == 0) {
            const uint32_t bar_q = bars + 8 * kBarQFull;
            uint32_t n = 0;       // ring entries produced so far (all items)
            bool ok = true;
            int q_item = 0;       // the last phase of bar_q that was armed: an item's Q tiles, or the end of the items
            int id = (int)blockIdx.x;
            for (uint32_t item = 0; ok; ++item) {
                if (item > 0) ok = wait_bar(bars + 8 * kBarQFree, (item - 1) & 1, ab, 50);
                if (!ok) break;
                if (id >= p.n_sched) {
                    item_slots[item & 1] = -1;
                    mbar_arrive(bar_q);
                    q_item = (int)item;
                    break;
                }
                const Item it = decode_item<kSplit>(id, p);
                const int j0 = kSplit ? it.j0 : 0, nj = kSplit ? it.nj : n_kv;
                if (item > 0) request_q(item & 1, id, it);
                q_item = (int)item;
                // K comes from the kernel before this one: up to here everything ran beside its end
                if (item == 0) {
                    if (p.k_made_before) grid_dependency_sync();
                    prefetch_tensormap(&tm_w);
                    prefetch_tensormap(&tm_s);
                }
                const int entries = item_entries(it, nj);
                for (int e = 0; e < entries && ok; ++e, ++n) {
                    const uint32_t slot = n % kStages;
                    if (n >= (uint32_t)kStages)
                        ok = wait_bar(bars + 8 * (kBarEmpty0 + slot), ((n / kStages) - 1) & 1, ab, 51);
                    if (!ok) break;
                    const uint32_t bar = bars + 8 * (kBarFull0 + slot);
                    const uint32_t dst = smem_base + kOffRing + slot * kTileBytes;
                    mbar_expect_tx(bar, kTileBytes);
                    const Entry en = item_entry(it, nj, e);
                    const int tb = it.b[en.tile], th = it.h[en.tile];
                    if (en.kind == kEntK || en.kind == kEntV) {
                        const CUtensorMap* tm = en.kind == kEntV ? &tm_v : &tm_k;
                        tma_load_4d(dst, tm, bar, 0, th, (j0 + en.j) * kTile, tb);
                        tma_load_4d(dst + kHalfBytes, tm, bar, 64, th, (j0 + en.j) * kTile, tb);
                    } else if (en.kind == kEntW) {
                        tma_load_2d(dst, &tm_w, bar, 0, th * kTile);
                        tma_load_2d(dst + kHalfBytes, &tm_w, bar, 64, th * kTile);
                    } else if (en.kind == kEntQRaw) {
                        tma_load_4d(dst, &tm_q, bar, 0, th, it.row0[en.tile], tb);
                        tma_load_4d(dst + kHalfBytes, &tm_q, bar, 64, th, it.row0[en.tile], tb);
                    } else {
                        tma_load_2d(dst, &tm_s, bar, 0, (tb * p.s.H + th) * kTile);
                        tma_load_2d(dst + kHalfBytes, &tm_s, bar, 64, (tb * p.s.H + th) * kTile);
                    }
                }
                if (!ok) break;
                // Every item is followed by one draw, so the launch makes n_sched of them: the last leaves the counter as it
                // was found, and the same launch may run again (a graph that is replayed).
                const uint32_t drawn = atomicAdd(p.sched_counter, 1u);
                if (drawn + 1 == (uint32_t)p.n_sched) *p.sched_counter = 0;
                id = (int)gridDim.x + (int)drawn;
            }
            // Do not leave the CTA while bulk copies into its shared memory are in flight.  Whatever became of the waits here: a
            // role that copies were for may give up after this one is through.
            drain_bar(bar_q, (uint32_t)q_item & 1);
            for (uint32_t m = (n > (uint32_t)kStages ? n - kStages : 0); m < n; ++m)
                drain_bar(bars + 8 * (kBarFull0 + m % kStages), (m / kStages) & 1);
        }
    } else if (warp == 9 || warp == 10) {
        // ---------------- MMA issuers: warp 9 drives query tile 0, warp 10 tile 1 ----------------
        // Both issuers walk the same sequence of ring entries and both release every entry (the empty
        // barriers count two arrivals), whether or not they read it.
        //
        // The serial chain of a tile -- S ready, softmax, P ready, P V and the next S -- sets the time of a
        // key iteration, so what an issuer adds to it counts.  (1) The whole warp walks the loop and one
        // elected lane issues: the 16 MMAs of an iteration are then issued in 770 clk and run back to back (1275
        // clk from P ready to S ready); issued by a single live lane they took 1125 to 1385, more the busier the
        // softmax warps were (presumably because a warp in uniform control flow can keep descriptors and
        // addresses in uniform registers; measured is the issue time only).  (2) The issuers take turns, 16 MMAs each: interleaved, both
        // tiles' MMAs end late and the two softmax groups fall into step (0.57 ms for L = 4680, 40 heads;
        // the turn the groups used to take in the exponential phase instead left the exponential unit idle
        // between them).  Key iteration 3790 -> 3310 clk; that shape 0.447 -> 0.423 ms per pass at full clocks,
        // 0.502 -> 0.479 under the power cap; 4680 queries against a cache of 18720 tokens, 12 heads: 0.548 -> 0.514.
        {
            const uint32_t lead = elect_one();
            const int t = __shfl_sync(0xffffffffu, warp - 9, 0);
            const uint32_t smem_base = __shfl_sync(0xffffffffu, smem_u32(smem), 0);
            const uint32_t bars = smem_base + kOffBars;
            const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);
            constexpr uint32_t idesc_qk = idesc_bf16(kTile, kTile, 0, 0);  // A, B K-major
            constexpr uint32_t idesc_pv = idesc_bf16(kTile, kTile, 0, 1);  // A in TMEM, B N-contiguous
            const uint32_t q_tile = smem_base + kOffQ + t * kTileBytes;
            const uint32_t s_col = tmem_base + t * kTile;
            const uint32_t o_col = tmem_base + 2 * kTile + t * kTile;
            const uint32_t bar_s = bars + 8 * (kBarSFull0 + t);
            const uint32_t bar_p = bars + 8 * (kBarPFull0 + t);

            // Matrix descriptors are built once: the high word is constant (stride between 8-row
            // groups, version, swizzle) and a k-step only adds to the 16-byte-unit start address.
            const uint32_t desc_hi = (uint32_t)(smem_desc_sw128(0, 0) >> 32);
            constexpr uint32_t kLboK = 1u << 16;                                // K-major: unused field
            constexpr uint32_t kLboMN = (uint32_t)(kHalfBytes >> 4) << 16;      // 64-column groups of V
            auto desc64 = [&](uint32_t lo) {
                uint64_t d;
                asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(desc_hi));
                return d;
            };
            // S_t (or U_t) = A_t * B^T with both operands K-major, 8 k-steps of 16
            auto issue_qk = [&](uint32_t a_tile, uint32_t b_tile) {
                const uint32_t a_lo = (a_tile >> 4) | kLboK, b_lo = (b_tile >> 4) | kLboK;
#pragma unroll
                for (int ks = 0; ks < 8; ++ks) {
                    const uint32_t koff = (uint32_t)(((ks >> 2) * kHalfBytes + (ks & 3) * 32) >> 4);
                    mma_ss_if(lead, s_col, desc64(a_lo + koff), desc64(b_lo + koff), idesc_qk, ks > 0);
                }
            };
            // O_t (+)= P_t * V with P in TMEM and V rows = contraction index, 8 k-steps of 16
            auto issue_pv = [&](uint32_t v_tile, bool accumulate) {
                const uint32_t v_lo = (v_tile >> 4) | kLboMN;
#pragma unroll
                for (int ks = 0; ks < 8; ++ks)
                    mma_ts_if(lead, o_col, s_col + ks * 8, desc64(v_lo + (uint32_t)(ks * (2048 >> 4))), idesc_pv,
                           (accumulate || ks > 0) ? 1u : 0u);
            };
            auto slot_addr = [&](uint32_t entry) { return smem_base + kOffRing + (entry % kStages) * kTileBytes; };
            auto wait_full = [&](uint32_t entry, int site) {
                return wait_bar_warp(bars + 8 * (kBarFull0 + entry % kStages), (entry / kStages) & 1, ab, site);
            };
            auto release = [&](uint32_t entry) { mma_commit_if(lead, bars + 8 * (kBarEmpty0 + entry % kStages)); };

            uint32_t cons = 0;        // ring entries consumed so far (all items)
            uint32_t p_cnt = 0;       // phases of bar_p consumed
            uint32_t qrot_cnt = 0, of_cnt = 0;
            uint32_t turn = 0;        // turns taken on the tensor pipe
            bool ok = true;
            for (uint32_t item = 0; ok; ++item) {
                ok = wait_bar_warp(bars + 8 * kBarQFull, item & 1, ab, 60);
                if (!ok) break;
                const int id = __shfl_sync(0xffffffffu, item_slots[item & 1], 0);
                if (id < 0) break;
                const Item it = decode_item<kSplit>(id, p);
                const int nj = kSplit ? it.nj : n_kv;   // key tiles of this item (a part walks its own range)
                const int ntile = it.ntile;
                const bool active = t < ntile;
                const bool shared = it.shared;
                // An entry both tiles read (K, V, W, S of a pair item) is released once by each
                // issuer; an entry only one tile reads is released twice by that tile's issuer
                // (the empty barriers always count two arrivals) and ignored by the other.
                auto release_mine = [&](uint32_t e, bool exclusive) {
                    release(e);
                    if (exclusive) release(e);
                };
                auto q_free = [&]() {
                    mma_commit_if(lead, bars + 8 * kBarQFree);
                    if (ntile == 1) mma_commit_if(lead, bars + 8 * kBarQFree);   // on behalf of the idle issuer
                };
                if (active) {
                    ok = wait_bar_warp(bars + 8 * (kBarQRot0 + t), qrot_cnt & 1, ab, 61);
                    ++qrot_cnt;
                    if (!ok) break;
                    // S_t(0) = Q~_t K_0^T
                    const uint32_t e_k = cons + (shared ? 0 : t);
                    ok = wait_full(e_k, 62);
                    if (!ok) break;
                    tc_fence_after();
                    issue_qk(q_tile, slot_addr(e_k));
                    mma_commit_if(lead, bar_s);
                    release_mine(e_k, !shared);
                    if (nj == 1) q_free();
                }
                cons += shared ? 1 : ntile;

                for (int j = 0; j < nj && ok; ++j) {
                    const bool last = j + 1 == nj;       // then the next "S" is the inter branch's Q W
                    const int per_tile = last ? 3 : 2;   // ragged item: V, K or W, [Qraw] per tile
                    const int group = shared ? (last ? 2 + ntile : 2) : per_tile * ntile;
                    if (active) {
                        const uint32_t e_v = shared ? cons : cons + per_tile * t;   // V_j
                        const uint32_t e_b = e_v + 1;                               // K_{j+1} or W
                        const uint32_t e_q = shared ? cons + 2 + t : e_v + 2;       // raw Q tile (last only)
                        ok = wait_full(e_v, 63);
                        if (ok) ok = wait_full(e_b, 66);
                        if (ok && last) ok = wait_full(e_q, 68);
                        if (!ok) break;
                        if (ntile == 2) {
                            ok = wait_bar_warp(bars + 8 * (kBarTurn0 + t), (t == 0) ? ((turn + 1) & 1) : (turn & 1), ab,
                                               24 + t);
                            ++turn;
                            if (!ok) break;
                        }
                        ok = wait_bar_warp(bar_p, p_cnt & 1, ab, 64 + t);
                        ++p_cnt;
                        if (!ok) break;
                        tc_fence_after();
                        issue_pv(slot_addr(e_v), j > 0);
                        issue_qk(last ? slot_addr(e_q) : q_tile, slot_addr(e_b));
                        mma_commit_if(lead, bar_s);
                        if (ntile == 2) mbar_arrive_if(lead, bars + 8 * (kBarTurn0 + (t ^ 1)));
                        release_mine(e_v, !shared);
                        release_mine(e_b, !shared);
                        if (last) release_mine(e_q, true);
                        if (j + 2 == nj) q_free();   // the last score MMA was the last use of Q~
                    }
                    cons += group;
                }
                if (!ok) break;
                // inter branch: O_t += Q''_t S
                if (active) {
                    const uint32_t e_s = cons + (shared ? 0 : t);
                    ok = wait_full(e_s, 69);
                    if (ok) ok = wait_bar_warp(bar_p, p_cnt & 1, ab, 70 + t);
                    ++p_cnt;
                    if (!ok) break;
                    tc_fence_after();
                    if constexpr (kElemGate) {
                        // per-channel gates: X = Q' S kept apart from O_t, 64 channels at a time into
                        // columns 64-127 of S_t (Q' sits in columns 0-63)
                        constexpr uint32_t idesc_x = idesc_bf16(kTile, 64, 0, 1);
                        for (int hv = 0; hv < 2 && ok; ++hv) {
                            if (hv == 1) {
                                ok = wait_bar_warp(bar_p, p_cnt & 1, ab, 72 + t);   // first half consumed
                                ++p_cnt;
                                if (!ok) break;
                                tc_fence_after();
                            }
                            const uint32_t x_lo = ((slot_addr(e_s) + hv * kHalfBytes) >> 4) | kLboMN;
#pragma unroll
                            for (int ks = 0; ks < 8; ++ks)
                                mma_ts_if(lead, s_col + 64, s_col + ks * 8, desc64(x_lo + (uint32_t)(ks * (2048 >> 4))), idesc_x,
                                       ks > 0 ? 1u : 0u);
                            mma_commit_if(lead, bar_s);
                        }
                        if (!ok) break;
                        release_mine(e_s, !shared);
                    } else {
                        issue_pv(slot_addr(e_s), true);
                        release_mine(e_s, !shared);
                        mma_commit_if(lead, bars + 8 * (kBarOFinal0 + t));
                        ++of_cnt;
                    }
                }
                cons += shared ? 1 : ntile;
            }
            (void)of_cnt;
            // tensor memory is freed below: none of this thread's MMAs may still be running, even if the softmax group gives up on
            // them after this
            mma_commit_if(lead, bars + 8 * (kBarDrain0 + t));
            drain_bar(bars + 8 * (kBarDrain0 + t), 0);
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 9) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

// ---------------------------------------------------------------------------------------------
// Token-sequential commit with per-token gates (Eq. 4 token by token), chunkwise, tensor cores.
// Notation as in the plain-FMA version: for a chunk of C = 64 tokens entering with state S_0,
//   U = U1 - W S_0,  S_C = g S_0 + Khat^T U,  U1 = T diag(beta) V',  W = T diag(beta g_{j-1}) K',
//   T = (I + A)^-1,  A_ji = beta_j (g_{j-1} / g_i) <K'_j, K'_i> (i < j),  Khat_i = (g / g_i) K'_i.
// tc_token_prepare_kernel: one CTA per 128-token tile = two chunks; 256 threads, two per token row
// (thread 0 also issues the copies and MMAs).  A tile is a chain of dependent stages, so two CTAs share an SM (96 KB of
// tiles and 256 TMEM columns each) and hide each other's latencies:
//   U_k = K W_k -> K' (bf16, over K);  U_v = V W_v -> diag(beta) V' (bf16, over V)        W_v replaces W_k
//   Gram matrix K' K'^T -> A (fp32, column by column, over W_v);  diag(beta g) K' over K'
//   T = (I + A)^-1 in place: the four 16 x 16 diagonal blocks of a chunk by forward substitution (thread =
//   column), then T21 = -T22 A21 T11 for blocks of 16 and of 32 (all threads)
//   T as a bf16 operand (over A): 128 x 128, zero off the chunks' blocks
//   W = T diag(beta g) K' and U1 = T diag(beta) V', T with both chunks' blocks on its diagonal (the zeros cost no MMA: with one per
//   chunk over all 128 rows, U1 had no columns of its own and waited for W's write-out) -> global: W, U1 (and Khat on the way) in
//   bf16, chunk decays g in fp32.
// 12 heads x 4680 tokens (444 tiles), inside the call: 66 us with one 128-thread CTA per SM, T by one 64-step
// substitution per column and row-wise stores -> 42 us; 40 heads 205 -> 112 (each alone).
// tc_token_scan_kernel: walks the chunks of a head in order (further down).
// ---------------------------------------------------------------------------------------------
constexpr int kTPOffK = 0;                         // raw K tile -> K' -> diag(beta g) K'
constexpr int kTPOffV = kTileBytes;                // raw V tile -> diag(beta) V'
constexpr int kTPOffW = 2 * kTileBytes;            // W_k; then W_v; then A -> T (2 x 64 x 68 fp32); then T (bf16)
constexpr int kTokC = 64;                          // tokens per chunk
constexpr int kLdA = kTokC + 4;                    // column stride of A: 16-byte aligned, columns spread over the banks
constexpr int kTPOffBars = kTPOffW + 2 * kTokC * kLdA * 4;
constexpr int kTPSmemBytes = kTPOffBars + 1024 + 1024 + 1024;   // barriers, gate scratch, alignment slack
constexpr int kTPThreads = 256;
static_assert(2 * kTokC * kLdA * 4 >= kTileBytes && kTPSmemBytes <= 115712, "two CTAs per SM");

enum TPBar : int { kTPBarLoadK = 0, kTPBarLoadV, kTPBarLoadW, kTPBarUk, kTPBarUv, kTPBarG, kTPBarW, kTPBarU1, kTPBarDrain, kTPNumBars };

struct TcTokenParams {
    Shape s;
    const uint4* rope_h;
    const float* alpha;        // [B, L, H] logits or nullptr
    const float* beta;
    __nv_bfloat16* w;          // [B, H, rows_pad, 128]
    __nv_bfloat16* kh;         // [B, H, rows_pad, 128]
    __nv_bfloat16* u1;         // [B, H, rows_pad, 128]
    float* gc;                 // [B, H, 2 * ntile]
    float* state;              // the walk reads it, the publishing kernel writes it and its bf16 copy
    __nv_bfloat16* state_bf16;
    float* next;               // [B, H, 2 runs - 1, 128, 128]: S after the walk (of the first run, then N and M of each further one), until it is published
    uint32_t* status;
    uint32_t spin_limit;
    uint32_t walk_limit;       // n > 0: the first wait of the walk's last CTA gives up after n - 1 polls (test hook)
    int ntile;                 // 128-token tiles; rows_pad = 128 * ntile
    int nchunk;                // ceil(L / 64): chunks the scan walks
    int runs, run_chunks;      // runs a head's chunks are cut into, and chunks of a run (the last one may be shorter)
    int decayed;               // prediction against alpha_j S_{j-1}
};

__global__ void __launch_bounds__(kTPThreads, 2)
tc_token_prepare_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                        const __grid_constant__ CUtensorMap tm_wk, const __grid_constant__ CUtensorMap tm_wv,
                        const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_u1,
                        const TcTokenParams p)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                               ~static_cast<uintptr_t>(1023));
    const uint32_t smem_base = smem_u32(smem);
    const uint32_t bars = smem_base + kTPOffBars;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + kTPOffBars + kTPNumBars * 8);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + kTPOffBars + kTPNumBars * 8 + 4);
    float* cl_s = reinterpret_cast<float*>(smem + kTPOffBars + 128);         // [128] log g_j (inclusive)
    float* wsum = reinterpret_cast<float*>(smem + kTPOffBars + 128 + 512);   // [8] warp totals
    float* ss_s = reinterpret_cast<float*>(smem + kTPOffBars + 1024);        // [2][128] sums of squares of the half rows
    const Abort ab{abort_flag, p.status, p.spin_limit};

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int tile = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
    const int L = p.s.L, H = p.s.H;
    // two threads per token row: warps w and w + 4 own the same 32 TMEM lanes and split the 128 columns
    const int r = (warp & 3) * 32 + lane;        // token row of the tile
    const int hf = warp >> 2;                    // which 64 of the 128 columns
    const int row = tile * kTile + r;            // this thread's token
    const int chunk = r >> 6, jj = r & 63;       // chunk of the tile, index in the chunk

    grid_dependency_sync();
    // the gates and the rotation table are asked for before anything else: behind the first copies and MMAs, which
    // keep the issuing warp, they held the whole CTA up by some 6 k of 44 k clk (12 heads x 4680 tokens 87.5 -> 83.1 us per
    // pass, together with W leaving under the product for U1)
    float alpha_logit = 0.0f, beta_logit = 0.0f;
    uint4 cs[8];
    if (row < L) {
        const size_t gi = ((size_t)b * L + row) * H + h;
        if (p.alpha != nullptr) alpha_logit = p.alpha[gi];
        if (p.beta != nullptr) beta_logit = p.beta[gi];
    }
    if (p.rope_h != nullptr) {
        const uint4* tab = p.rope_h + ((size_t)(row >> 5) * 16 + hf * 8) * 32 + (row & 31);
#pragma unroll
        for (int c = 0; c < 8; ++c) cs[c] = tab[c * 32];
    }
    if (tid == 0) {
        for (int i = 0; i < kTPNumBars; ++i) mbar_init(bars + 8 * i, 1);
        *abort_flag = 0;
        fence_barrier_init();
        fence_proxy_async_smem();
        const uint32_t bar_k = bars + 8 * kTPBarLoadK, bar_v = bars + 8 * kTPBarLoadV;
        mbar_expect_tx(bar_k, 2 * kTileBytes);
        mbar_expect_tx(bar_v, kTileBytes);
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            tma_load_2d(smem_base + kTPOffW + half * kHalfBytes, &tm_wk, bar_k, half * 64, h * kTile);
            tma_load_4d(smem_base + kTPOffK + half * kHalfBytes, &tm_k, bar_k, half * 64, h, tile * kTile, b);
        }
#pragma unroll
        for (int half = 0; half < 2; ++half)
            tma_load_4d(smem_base + kTPOffV + half * kHalfBytes, &tm_v, bar_v, half * 64, h, tile * kTile, b);
    }
    if (warp == 0) {
        tmem_alloc(smem_u32(tmem_slot), 256);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    const uint32_t lane_base = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);

    constexpr uint32_t kLboK = 1u << 16;
    constexpr uint32_t kLboMN = (uint32_t)(kHalfBytes >> 4) << 16;
    const uint32_t desc_hi = (uint32_t)(smem_desc_sw128(0, 0) >> 32);
    auto desc64 = [&](uint32_t lo) {
        uint64_t d;
        asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(desc_hi));
        return d;
    };
    constexpr uint32_t idesc_kk = idesc_bf16(kTile, kTile, 0, 0);   // both operands d-major
    constexpr uint32_t idesc_kn = idesc_bf16(kTile, kTile, 0, 1);   // A K-major, B rows = contraction index
    auto koff_k = [](int ks) { return (uint32_t)(((ks >> 2) * kHalfBytes + (ks & 3) * 32) >> 4); };
    const bool issuer = tid == 0;
    bool ok = true;                              // the issuer's waits
    bool alive = true;                           // the row threads' waits
    bool w_loaded = false;
    // D[128 x 128] = A[128 x 128] B^T, both d-major
    auto issue_kk = [&](uint32_t col, int a_off, int b_off) {
        const uint32_t a_lo = ((smem_base + a_off) >> 4) | kLboK, b_lo = ((smem_base + b_off) >> 4) | kLboK;
#pragma unroll
        for (int ks = 0; ks < 8; ++ks)
            mma_ss(tmem_base + col, desc64(a_lo + koff_k(ks)), desc64(b_lo + koff_k(ks)), idesc_kk, ks > 0);
    };
    // D[128 x 128] = T (both chunks' blocks on its diagonal) times a tile, tokens contracted
    auto issue_t = [&](uint32_t col, int b_off) {
        const uint32_t t_lo = ((smem_base + kTPOffW) >> 4) | kLboK, b_lo = ((smem_base + b_off) >> 4) | kLboMN;
#pragma unroll
        for (int ks = 0; ks < 8; ++ks)
            mma_ss(tmem_base + col, desc64(t_lo + koff_k(ks)), desc64(b_lo + (uint32_t)(ks * (2048 >> 4))), idesc_kn, ks > 0);
    };

    // ---- gates: log alpha_j, beta_j, cumulative decay within the chunk (tokens past L: 1 and 0)
    float la = 0.0f, be = 0.0f, cl = 0.0f;
    if (row < L) {
        if (p.alpha != nullptr) {
            const float x = alpha_logit;
            la = x >= 0.0f ? -log1pf(expf(-x)) : x - log1pf(expf(x));
        }
        be = p.beta != nullptr ? 1.0f / (1.0f + expf(-beta_logit)) : 1.0f;
    }
    cl = la;   // inclusive scan over the 64 tokens of the chunk (two warps)
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const float up = __shfl_up_sync(0xffffffffu, cl, off);
        if (lane >= off) cl += up;
    }
    if (lane == 31) wsum[warp] = cl;
    __syncthreads();
    if (warp & 1) cl += wsum[warp - 1];
    if (hf == 0) cl_s[r] = cl;
    __syncthreads();
    if (issuer) {
        // ---- U_k = K W_phi_k -> columns 0-127
        ok = wait_bar(bars + 8 * kTPBarLoadK, 0, ab, 90);
        if (ok) {
            tc_fence_after();
            issue_kk(0, kTPOffK, kTPOffW);
            mma_commit(bars + 8 * kTPBarUk);
        }
    }

    const float cl_total = cl_s[chunk * kTokC + kTokC - 1];
    const float cl_excl = cl - la;
    // log of the factor on K'_j S_0: g_{j-1} for Eq. 4 as printed, g_j when the token's prediction is made
    // against the state after its own forget gate
    const float cl_pred = p.decayed ? cl : cl_excl;

    // 32 columns of this thread's half row (piece q of 2) into a swizzled tile, times f
    auto put32_at = [&](int off, int half, int q, const uint32_t (&y)[32], float f) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            uint32_t w[4];
#pragma unroll
            for (int m = 0; m < 4; ++m)
                w[m] = pack_bf16(__uint_as_float(y[c * 8 + 2 * m]) * f, __uint_as_float(y[c * 8 + 2 * m + 1]) * f);
            *reinterpret_cast<uint4*>(smem + off + half * kHalfBytes + r * 128 + (((q * 4 + c) ^ (r & 7)) << 4)) =
                make_uint4(w[0], w[1], w[2], w[3]);
        }
    };
    auto put32 = [&](int off, int q, const uint32_t (&y)[32], float f) { put32_at(off, hf, q, y, f); };
    alive = wait_bar(bars + 8 * kTPBarUk, 0, ab, 96);
    if (issuer && ok && alive) {
        // the value map takes the key map's place while the rows of K' are worked out
        const uint32_t bar = bars + 8 * kTPBarLoadW;
        mbar_expect_tx(bar, kTileBytes);
        tma_load_2d(smem_base + kTPOffW, &tm_wv, bar, 0, h * kTile);
        tma_load_2d(smem_base + kTPOffW + kHalfBytes, &tm_wv, bar, 64, h * kTile);
        w_loaded = true;
    }
    float ss4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    if (alive) {
        tc_fence_after();
        // ---- K' = L2Norm(RoPE(U_k)): the norm over the whole row first (a rotation leaves it as it is; half of it by each of
        // the row's threads: 40 heads x 4680 tokens 202.7 -> 200.6 us, 12 heads 70.8 -> 70.5), then
        // this thread's half, 32 columns at a time (with whole half rows in registers the kernel spilled at two
        // CTAs per SM: 4.5 k clk for this pass against 1.5 k): K' for the Gram matrix, Khat to global memory,
        // and K' in fp32 back to the columns of U_k for diag(beta g) K'
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            uint32_t y[32];
            tmem_ld32(lane_base + hf * 64 + q * 32, y);
            tmem_wait_ld();
#pragma unroll
            for (int c = 0; c < 32; ++c) ss4[c & 3] = fmaf(__uint_as_float(y[c]), __uint_as_float(y[c]), ss4[c & 3]);
        }
    }
    ss_s[hf * kTile + r] = (ss4[0] + ss4[1]) + (ss4[2] + ss4[3]);
    __syncthreads();
    if (alive) {
        const float f = rsqrtf(ss_s[r] + ss_s[kTile + r] + p.s.eps);
        const float f_kh = expf(cl_total - cl);
        // ---- U_v = V W_phi_v -> columns 128-255: after the first half of this pass if both operands have landed, so that the
        // product is there when the second half is done (5 x 700 tokens 22.3 -> 21.8 us, 12 heads x 4680 71.3 -> 70.8; waiting for
        // them there held the issuing warp's own rows up: 72.0)
        auto issue_uv = [&]() {
            tc_fence_after();
            issue_kk(kTile, kTPOffV, kTPOffW);
            mma_commit(bars + 8 * kTPBarUv);
        };
        bool uv_sent = false;
        __nv_bfloat16* kh = p.kh + ((((size_t)b * H + h) * p.ntile + tile) * kTile + r) * kTile + hf * 64;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            uint32_t y[32];
            tmem_ld32(lane_base + hf * 64 + q * 32, y);
            tmem_wait_ld();
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint4 v = p.rope_h != nullptr ? cs[q * 4 + c] : make_uint4(0x3C00u, 0x3C00u, 0x3C00u, 0x3C00u);   // cos 1, sin 0
                const uint32_t h2[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    float cc, s1;
                    unpack_cs(h2[m], cc, s1);
                    const float x0 = __uint_as_float(y[c * 8 + 2 * m]) * f, x1 = __uint_as_float(y[c * 8 + 2 * m + 1]) * f;
                    y[c * 8 + 2 * m] = __float_as_uint(x0 * cc - x1 * s1);
                    y[c * 8 + 2 * m + 1] = __float_as_uint(x0 * s1 + x1 * cc);
                }
            }
            if (q == 0 && issuer && ok && mbar_test_wait(bars + 8 * kTPBarLoadW, 0) && mbar_test_wait(bars + 8 * kTPBarLoadV, 0)) {
                issue_uv();
                uv_sent = true;
            }
            tmem_st32(lane_base + hf * 64 + q * 32, y);
            put32(kTPOffK, q, y, 1.0f);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                uint32_t w[8];
#pragma unroll
                for (int m = 0; m < 8; ++m)
                    w[m] = pack_bf16(__uint_as_float(y[e * 16 + 2 * m]) * f_kh, __uint_as_float(y[e * 16 + 2 * m + 1]) * f_kh);
                asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(kh + q * 32 + e * 16),
                             "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                             : "memory");
            }
        }
        tmem_wait_st();
        if (issuer && ok && !uv_sent) {
            ok = wait_bar(bars + 8 * kTPBarLoadW, 0, ab, 94);
            if (ok) ok = wait_bar(bars + 8 * kTPBarLoadV, 0, ab, 95);
            if (ok) issue_uv();
        }
        alive = wait_bar(bars + 8 * kTPBarUv, 0, ab, 97);
        if (alive) {
            tc_fence_after();
            // ---- diag(beta) V'
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                uint32_t y[32];
                tmem_ld32(lane_base + kTile + hf * 64 + q * 32, y);
                tmem_wait_ld();
                put32(kTPOffV, q, y, be);
            }
        }
    }
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();

    // ---- Gram matrix K' K'^T -> columns 128-255 (row = token j, column = token i)
    if (issuer && ok && !*abort_flag) {
        tc_fence_after();
        issue_kk(kTile, kTPOffK, kTPOffK);
        mma_commit(bars + 8 * kTPBarG);
    }
    float* As = reinterpret_cast<float*>(smem + kTPOffW);   // the maps are dead: U_k, U_v are complete
    alive = alive && wait_bar(bars + 8 * kTPBarG, 0, ab, 92);
    if (alive) {
        tc_fence_after();
        // this token's row of A: the columns of its own chunk, strictly below the diagonal (zero elsewhere),
        // stored column by column (a warp's 32 rows side by side).  All values before the first store: the
        // compiler may not move the reads of cl_s across stores to shared memory.
        uint32_t g[32];
        tmem_ld32(lane_base + kTile + chunk * kTokC + hf * 32, g);
        tmem_wait_ld();
        const float* cl_c = cl_s + chunk * kTokC + hf * 32;
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            float x = be * __expf(cl_pred - cl_c[i]) * __uint_as_float(g[i]);
            // worked out in any case: with a branch round each exponential this pass took 2.1 k clk, now 0.8 k (2 heads x 4680
            // tokens 37.6 -> 37.2 us, 12 heads 71.8 -> 71.3, 5 x 700 22.7 -> 22.3)
            asm volatile("" : "+f"(x));
            g[i] = hf * 32 + i < jj ? __float_as_uint(x) : 0u;
        }
        float* a_out = As + (chunk * kTokC + hf * 32) * kLdA + jj;
#pragma unroll
        for (int i = 0; i < 32; ++i) a_out[i * kLdA] = __uint_as_float(g[i]);
    }
    tc_fence_before();
    __syncthreads();
    // ---- T = (I + A)^-1, in place (element (i, j) of chunk c at X[(c * 64 + j) * kLdA + i])
    {
        // diagonal blocks: thread = (chunk, block, column) for the first 128 threads
        const int o = (tid >> 4 & 3) * 16, cc = tid & 15;
        float* Xd = As + ((tid >> 6) * kTokC + o) * kLdA + o;
        float t[16];
        if (tid < 128) {
#pragma unroll
            for (int i = 0; i < 16; ++i) t[i] = i == cc ? 1.0f : 0.0f;
#pragma unroll
            for (int j = 0; j < 15; ++j) {
                // as soon as t_j is known it is taken out of all later rows: a step is one FMA deep
#pragma unroll
                for (int i4 = (j + 1) / 4; i4 < 4; ++i4) {
                    const float4 a4 = *reinterpret_cast<const float4*>(Xd + j * kLdA + i4 * 4);
                    const float av[4] = {a4.x, a4.y, a4.z, a4.w};
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (i4 * 4 + k > j) t[i4 * 4 + k] = fmaf(-av[k], t[j], t[i4 * 4 + k]);
                }
            }
        } else if (alive) {
            // the other four warps meanwhile: diag(beta g) K' replaces K', which the Gram matrix was the last to read
            const float f_w = be * expf(cl_pred);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint32_t y[32];
                tmem_ld32(lane_base + q * 32, y);
                tmem_wait_ld();
                put32_at(kTPOffK, q >> 1, q & 1, y, f_w);
            }
        }
        __syncthreads();
        if (tid < 128) {
#pragma unroll
            for (int i4 = 0; i4 < 4; ++i4)
                *reinterpret_cast<float4*>(Xd + cc * kLdA + i4 * 4) = make_float4(t[i4 * 4], t[i4 * 4 + 1], t[i4 * 4 + 2], t[i4 * 4 + 3]);
        }
        __syncthreads();
        // out(i, j) = sign * sum over k0 <= k < k1 of P(i, k) Q(k, j) for i = i0 .. i0 + 3 and j = j0, j0 + JS ..: each operand given
        // by its first element; i is contiguous in P and out, k in Q.  Two lanes (xor 1 << SB) share these outputs, taking every
        // second group of four k; each ends up with half of the columns.  What binds it is the shared memory, 16 bytes
        // per thread and load, of which a wider block needs fewer per FMA, and the chain behind one load, which the split of k
        // halves; only the k where the triangular operand is not zero are walked (the same for a warp).
        // The chunks' warps take their shares in opposite order, since warps w and w + 4 issue from the same quarter of the SM.
        // Products 6.9 k of a CTA's 31 k clk with one row per thread and all k, 4.8 k with four rows and the triangles, 4.3 k so
        // (commit_tokens of 12 heads x 4680 tokens 76.4 -> 73.1 -> 71.8 us, of 40 220 -> 206.6 -> 203.0; the last step together with the
        // diagonal's idle warps and U1 under W, below).
        auto product = [&](auto nj_tag, auto js_tag, auto sb_tag, const float* P, const float* Q, float* out, float sign, int i0, int j0, int k0, int k1) {
            constexpr int NJ = decltype(nj_tag)::value, JS = decltype(js_tag)::value, SB = decltype(sb_tag)::value;
            const bool second = (lane >> SB & 1) != 0;
            float acc[NJ][4] = {};
#pragma unroll 2
            for (int k4 = k0 + (second ? 4 : 0); k4 < k1; k4 += 8) {
                float4 pv[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) pv[k] = *reinterpret_cast<const float4*>(P + (k4 + k) * kLdA + i0);
#pragma unroll
                for (int j = 0; j < NJ; ++j) {
                    const float4 q = *reinterpret_cast<const float4*>(Q + (j0 + j * JS) * kLdA + k4);
                    acc[j][0] = fmaf(pv[0].x, q.x, fmaf(pv[1].x, q.y, fmaf(pv[2].x, q.z, fmaf(pv[3].x, q.w, acc[j][0]))));
                    acc[j][1] = fmaf(pv[0].y, q.x, fmaf(pv[1].y, q.y, fmaf(pv[2].y, q.z, fmaf(pv[3].y, q.w, acc[j][1]))));
                    acc[j][2] = fmaf(pv[0].z, q.x, fmaf(pv[1].z, q.y, fmaf(pv[2].z, q.z, fmaf(pv[3].z, q.w, acc[j][2]))));
                    acc[j][3] = fmaf(pv[0].w, q.x, fmaf(pv[1].w, q.y, fmaf(pv[2].w, q.z, fmaf(pv[3].w, q.w, acc[j][3]))));
                }
            }
#pragma unroll
            for (int j = 0; j < NJ / 2; ++j) {
                float y[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float give = second ? acc[j][i] : acc[NJ / 2 + j][i], keep = second ? acc[NJ / 2 + j][i] : acc[j][i];
                    y[i] = sign * (keep + __shfl_xor_sync(0xffffffffu, give, 1 << SB));
                }
                *reinterpret_cast<float4*>(out + (j0 + (j + (second ? NJ / 2 : 0)) * JS) * kLdA + i0) = make_float4(y[0], y[1], y[2], y[3]);
            }
        };
        const int pw = (warp & 3) ^ (tid >= 128 ? 3 : 0);   // four warps per chunk
        float* X = As + (tid >> 7) * kTokC * kLdA;
        {
            // blocks of 16: rows 32 m + 16 .., columns 32 m ..; the intermediate A21 T11 goes to the unused
            // rows 0-15 of columns 32 + 16 m ..  Two warps per m: of columns 0-7 and 8-15 first, then of rows 0-7 and 8-15
            const int m = pw >> 1, w = pw & 1;
            float* low = X + (m * 32) * kLdA + m * 32 + 16;
            float* tmp = X + (32 + m * 16) * kLdA;
            const auto two = std::integral_constant<int, 2>();
            product(two, std::integral_constant<int, 1>(), two, low, X + (m * 32) * kLdA + m * 32, tmp, 1.0f, (lane & 3) * 4, w * 8 + (lane >> 3) * 2, w * 8, 16);
            __syncthreads();
            product(two, std::integral_constant<int, 8>(), std::integral_constant<int, 3>(), X + (m * 32 + 16) * kLdA + m * 32 + 16, tmp, low, -1.0f,
                    w * 8 + (lane >> 4) * 4, lane & 7, 0, w * 8 + 8);
            __syncthreads();
        }
        {
            // blocks of 32: rows 32 .., columns 0 ..; the intermediate in rows 0-31 of columns 32 ..  Four warps: of eight columns
            // each first, then of eight rows each
            float* low = X + 32;
            float* tmp = X + 32 * kLdA;
            const auto four = std::integral_constant<int, 4>();
            const auto bit3 = std::integral_constant<int, 3>();
            product(four, std::integral_constant<int, 1>(), bit3, low, X, tmp, 1.0f, (lane & 7) * 4, pw * 8 + (lane >> 4) * 4, pw * 8, 32);
            __syncthreads();
            product(four, std::integral_constant<int, 8>(), bit3, X + 32 * kLdA + 32, tmp, low, -1.0f, pw * 8 + (lane >> 4) * 4, lane & 7, 0, pw * 8 + 8);
            __syncthreads();
        }
        // T as a K-major swizzled operand (row = token, 64 columns of the row's own chunk, zeros in the other's), over the fp32 matrix
        uint4 tv[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int c16 = hf * 4 + q;
            uint32_t w[4];
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const int j = c16 * 8 + 2 * m;
                const float lo = As[(chunk * kTokC + j) * kLdA + jj], hi = As[(chunk * kTokC + j + 1) * kLdA + jj];
                w[m] = pack_bf16(j <= jj ? lo : 0.0f, j + 1 <= jj ? hi : 0.0f);
            }
            tv[q] = make_uint4(w[0], w[1], w[2], w[3]);
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint8_t* piece = smem + kTPOffW + r * 128 + (((hf * 4 + q) ^ (r & 7)) << 4);
            *reinterpret_cast<uint4*>(piece + chunk * kHalfBytes) = tv[q];
            *reinterpret_cast<uint4*>(piece + (1 - chunk) * kHalfBytes) = make_uint4(0, 0, 0, 0);
        }
    }
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();

    // ---- W = T diag(beta g) K' -> columns 0-127, U1 = T diag(beta) V' -> columns 128-255, on its way under W's write-out
    if (issuer && ok && !*abort_flag) {
        tc_fence_after();
        issue_t(0, kTPOffK);
        mma_commit(bars + 8 * kTPBarW);
        issue_t(kTile, kTPOffV);
        mma_commit(bars + 8 * kTPBarU1);
    }
#pragma unroll 1
    for (int u = 0; u < 2; ++u) {
        alive = alive && wait_bar(bars + 8 * (u == 0 ? kTPBarW : kTPBarU1), 0, ab, 93);
        if (alive) {
            tc_fence_after();
            // staged in the tile that this product was the last to read
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                uint32_t y[32];
                tmem_ld32(lane_base + u * kTile + hf * 64 + q * 32, y);
                tmem_wait_ld();
                put32(u == 0 ? kTPOffK : kTPOffV, q, y, 1.0f);
            }
        }
        fence_proxy_async_smem();
        __syncthreads();
        // ---- it leaves as a whole tile
        if (issuer && ok && alive && !*abort_flag) {
            const int r0 = (int)((((size_t)b * H + h) * p.ntile + tile) * kTile);
#pragma unroll
            for (int half = 0; half < 2; ++half)
                tma_store_2d(u == 0 ? &tm_w : &tm_u1, smem_base + (u == 0 ? kTPOffK : kTPOffV) + half * kHalfBytes, half * 64, r0);
        }
    }
    if (issuer) tma_store_wait_read();   // (whatever went out has been read)
    if (hf == 0 && alive && jj == kTokC - 1)
        p.gc[(((size_t)b * H + h) * p.ntile + tile) * 2 + chunk] = expf(cl_total);
    if (issuer && (!ok || *abort_flag)) {
        drain_bar(bars + 8 * kTPBarLoadK, 0);   // no bulk copy left in flight
        drain_bar(bars + 8 * kTPBarLoadV, 0);
        if (w_loaded) drain_bar(bars + 8 * kTPBarLoadW, 0);
        mma_commit(bars + 8 * kTPBarDrain);     // and no MMA still writing tensor memory
        drain_bar(bars + 8 * kTPBarDrain, 0);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 256);
    }
}

// tc_token_scan_kernel: the ordered walk over the chunks.  The columns of S never mix (U = U1 - W S and
// S <- g S + Khat^T U act on each value column alone), so a head's 128 columns are cut into slabs of 16, each
// walked by a group of four warps; a CTA holds kSlabs of them and the W, Khat and U1 tiles they share.
// The walk is a chain of ceil(L / 64) dependent chunks: what counts is the latency of one, not throughput.
// Everything is kept transposed (row = value column e), so that the warp-level tensor instruction
// hands every result on in the layout the next product needs:
//   U^T[16 x 64]  = U1^T - S^T W^T     A = S^T (bf16, 4 KB of shared memory), B = W as it lies; warp w: 16 tokens
//   S^T[16 x 128] = g S^T + U^T Khat   A = U^T (bf16, 2 KB of shared memory), B = Khat;         warp w: 32 keys d
// The fp32 state stays in registers for the whole walk (16 per thread).  Per chunk a warp runs 16 + 16
// instructions in four independent chains each and meets its group twice (named barriers, 128 threads);
// the B fragments of the next chunk are fetched while this chunk's products run.  A fifth warp per CTA
// streams the tiles through a TMA ring.
// Few heads leave SMs idle; kRuns cuts the chunks of a head into runs that are walked side by side.  What a run does to
// the state it is entered with is S -> M S + N: N is the walk from the zero state, M the walk from the identity without
// U1, so a further run has 256 columns instead of 128; tc_token_join_kernel puts the runs together.  Its error against 64 bits
// is that of one walk (rel. 2-norm 4.1e-3 for both at 12 x 4680, ratios of 0.93 to 1.00 with other gates, keys of a common
// direction, few key directions, a state that fits the block); only where tokens write next to nothing and both are at 1e-5
// (rates of 5e-5) is it up to 3 times the larger.  Not kept: the part of M's diagonal that its bf16 operand lacks added apart
// (that ratio 2.7, and 71.2 -> 76.8 us).  (One group of four
// warps for two slabs, so that both use a B fragment that was read once: 78.4 us at 12 heads x 4680 tokens instead of 76.4.)
// 12 heads x 4680 tokens, inside the call: 162 us with one CTA per head and the
// state in TMEM (two MMAs, two passes through registers, four CTA-wide meetings per chunk) -> 46 us (1.2 k clk per
// chunk; the 34 KB per chunk and SM that come from L2 are about 0.65 k of that).
constexpr int kChunkHalf = kTokC * 128;              // bytes of a 64-row, 64-column box
constexpr int kScanLdS = kTile + 8, kScanLdU = kTokC + 8;   // padded rows: conflict-free 8 x 8 loads
constexpr int kScanSlab = 16;
constexpr int kScanMaxStages = 6;
// kSlabs slabs per CTA; kShared: two CTAs share an SM (two stages each, fragments fetched when needed)
template <int kSlabs, bool kShared>
struct ScanCfg {
    static constexpr int kStages = kShared ? 2 : kSlabs == 1 ? 6 : 5;
    static constexpr int kStageBytes = 4 * kChunkHalf + kSlabs * kTokC * kScanSlab * 2;
    static constexpr int kOffS = kStages * kStageBytes;
    static constexpr int kOffBars = kOffS + kSlabs * kScanSlab * (kScanLdS + kScanLdU) * 2;
    static constexpr int kSmemBytes = kOffBars + 2 * kScanMaxStages * 8 + 8 + 1024;
    static constexpr int kThreads = kSlabs * 128 + 32;
    static_assert(kSmemBytes <= (kShared ? 115712 : 232448), "shared memory");
};

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
                 "{%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

template <int kSlabs, bool kShared, bool kRuns>
__global__ void __launch_bounds__(kSlabs * 128 + 32, kShared ? 2 : 1)
tc_token_scan_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_kh,
                     const __grid_constant__ CUtensorMap tm_u1, const TcTokenParams p)
{
    using Cfg = ScanCfg<kSlabs, kShared>;
    constexpr int kS = Cfg::kStages;
    constexpr uint32_t kStageBytes = (uint32_t)Cfg::kStageBytes;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                               ~static_cast<uintptr_t>(1023));
    const uint32_t smem_base = smem_u32(smem);
    const uint32_t bar_full = smem_base + Cfg::kOffBars;
    const uint32_t bar_free = bar_full + 8 * kScanMaxStages;
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + Cfg::kOffBars + 16 * kScanMaxStages);
    const Abort ab{abort_flag, p.status, p.spin_limit};

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int h = blockIdx.y, b = blockIdx.z;
    const size_t bh = (size_t)b * p.s.H + h;
    // first value column of this CTA; the run it walks, and whether these are columns of M
    int e0 = blockIdx.x * kSlabs * kScanSlab, run = 0;
    bool is_m = false;
    if (kRuns && e0 >= kTile) {
        run = 1 + (e0 - kTile) / (2 * kTile);
        e0 = (e0 - kTile) % (2 * kTile);
        is_m = e0 >= kTile;
        e0 %= kTile;
    }
    const int chunk0 = kRuns ? run * p.run_chunks : 0;
    const int nchunk = kRuns ? min(p.run_chunks, p.nchunk - chunk0) : p.nchunk;

    if (tid == 0) {
        for (int i = 0; i < kS; ++i) {
            mbar_init(bar_full + 8 * i, 1);
            mbar_init(bar_free + 8 * i, kSlabs * 4);
        }
        *abort_flag = 0;
        fence_barrier_init();
        fence_proxy_async_smem();
    }
    grid_dependency_sync();
    // (one answer for the whole CTA) after an error the chunk factors are not all there, and nothing is published
    if (__syncthreads_or(*reinterpret_cast<volatile uint32_t*>(p.status + kStatusError) != 0u)) return;

    if (warp == kSlabs * 4) {
        // ---------------- TMA producer ----------------
        if (lane == 0) {
            const int r0 = (int)(bh * p.ntile * kTile) + chunk0 * kTokC;
            bool ok = true;
            int c = 0;
            for (; c < nchunk; ++c) {
                const int s = c % kS;
                if (c >= kS) ok = wait_bar(bar_free + 8 * s, (uint32_t)(c / kS - 1) & 1u, ab, 100);
                if (!ok) break;
                const uint32_t bar = bar_full + 8 * s, dst = smem_base + s * kStageBytes;
                mbar_expect_tx(bar, kStageBytes);
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    tma_load_2d(dst + half * kChunkHalf, &tm_w, bar, half * 64, r0 + c * kTokC);
                    tma_load_2d(dst + (2 + half) * kChunkHalf, &tm_kh, bar, half * 64, r0 + c * kTokC);
                }
                tma_load_2d(dst + 4 * kChunkHalf, &tm_u1, bar, e0, r0 + c * kTokC);
            }
            // no bulk copy may be in flight into this CTA's shared memory when it ends, whatever the walkers do
            for (int m = (c > kS ? c - kS : 0); m < c; ++m) drain_bar(bar_full + 8 * (m % kS), (uint32_t)(m / kS) & 1u);
        }
        return;
    }

    // ---------------- the walk: slab `slab` of this CTA, warp wq of its four ----------------
    const int slab = warp >> 2, wq = warp & 3;
    const int mi = lane >> 3, mr = lane & 7;             // 8 x 8 block and row this lane addresses in a load
    const int ge = lane >> 2, gk = (lane & 3) * 2;       // fragment row (value column) and column pair
    __nv_bfloat16* s_s = reinterpret_cast<__nv_bfloat16*>(smem + Cfg::kOffS) + slab * kScanSlab * (kScanLdS + kScanLdU);
    __nv_bfloat16* u_s = s_s + kScanSlab * kScanLdS;
    const uint32_t a_s = smem_u32(s_s) + (uint32_t)((((mi & 1) * 8 + mr) * kScanLdS + (mi >> 1) * 8) * 2);
    const uint32_t a_u = smem_u32(u_s) + (uint32_t)((((mi & 1) * 8 + mr) * kScanLdU + (mi >> 1) * 8) * 2);
    // offsets inside a stage (128-byte swizzle: the 16-byte piece index is xored with the row)
    const uint32_t w_row = (uint32_t)(wq * 16 + (mi >> 1) * 8 + mr);
    const uint32_t u1_off = 4 * kChunkHalf + (w_row * kSlabs * kScanSlab + (uint32_t)(slab * kScanSlab + (mi & 1) * 8)) * 2;
    auto group_sync = [&]() { asm volatile("bar.sync %0, 128;" ::"r"(slab + 1) : "memory"); };

    // state: st[n][0..1] = S[d][e], S[d + 1][e], st[n][2..3] the same for e + 8, d = 32 wq + 8 n + gk
    float st[4][4];
    float* srow = p.state + (bh * kTile + wq * 32 + gk) * kTile + e0 + slab * kScanSlab + ge;
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            if (run == 0) st[n][x] = srow[(size_t)(n * 8 + (x & 1)) * kTile + (x >> 1) * 8];
            else st[n][x] = is_m && wq * 32 + gk + n * 8 + (x & 1) == e0 + slab * kScanSlab + ge + (x >> 1) * 8 ? 1.0f : 0.0f;
        }
    auto put_s = [&]() {
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            *reinterpret_cast<uint32_t*>(s_s + ge * kScanLdS + wq * 32 + n * 8 + gk) = pack_bf16(st[n][0], st[n][1]);
            *reinterpret_cast<uint32_t*>(s_s + (ge + 8) * kScanLdS + wq * 32 + n * 8 + gk) = pack_bf16(st[n][2], st[n][3]);
        }
    };
    put_s();
    const float* gc = p.gc + bh * 2 * p.ntile + chunk0;
    const uint32_t u1_mask = is_m ? 0u : 0xFFFFFFFFu;
    float g_cur = lane < nchunk ? gc[lane] : 1.0f;   // decays of 32 chunks, one per lane

    bool dead = false;
    // On a wait that expires the warp goes on without waiting: the barriers of the group keep their
    // counts, the loop is finite, and the recorded error keeps the result from being published.
    auto landed = [&](int c) {
        if (!dead) dead = !wait_bar_warp(bar_full + 8 * (c % kS), (uint32_t)(c / kS) & 1u, ab, 101);
    };
    auto release = [&](int c) {
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_free + 8 * (c % kS));
    };
    auto stage = [&](int c) { return smem_base + (uint32_t)(c % kS) * kStageBytes; };
    auto load_w = [&](uint32_t (&f)[4], uint32_t base, int ks) {
        ldsm4(f, base + (uint32_t)(ks >> 2) * kChunkHalf + w_row * 128 + ((((uint32_t)(ks & 3) * 2 + (mi & 1)) ^ (w_row & 7)) << 4));
    };
    auto load_k = [&](uint32_t (&f)[4], uint32_t base, int ks, int j) {
        const uint32_t row = (uint32_t)(ks * 16 + (mi & 1) * 8 + mr);
        ldsm4t(f, base + (uint32_t)(2 + (wq >> 1)) * kChunkHalf + row * 128 +
                      ((((uint32_t)(wq & 1) * 4 + j * 2 + (mi >> 1)) ^ (row & 7)) << 4));
    };
    // fragments of the chunk at hand; kShared: filled just before their use instead of a chunk ahead
    uint32_t wf[kShared ? 1 : 8][4], kf[kShared ? 1 : 4][2][4], uf[4];
    auto load_all_w = [&](int c) {
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) load_w(wf[kShared ? 0 : ks], stage(c), ks);
    };
    auto load_all_k = [&](int c) {
#pragma unroll
        for (int ks = 0; ks < 4; ++ks)
#pragma unroll
            for (int j = 0; j < 2; ++j) load_k(kf[kShared ? 0 : ks][j], stage(c), ks, j);
        ldsm4t(uf, stage(c) + u1_off);
    };

    // (a wait of its own before the walk: a limit that differs between CTAs, read at every wait, cost the walk 2.8 us of 46)
    if (p.walk_limit != 0u && blockIdx.x + 1 == gridDim.x && blockIdx.y + 1 == gridDim.y && blockIdx.z + 1 == gridDim.z)
        dead = !wait_bar_warp(bar_full, 0, Abort{abort_flag, p.status, p.walk_limit - 1}, 101);
    if (!kShared) {
        landed(0);
        load_all_w(0);
        load_all_k(0);
        release(0);
    }
    group_sync();
    for (int c = 0; c < nchunk; ++c) {
        const bool more = c + 1 < nchunk;
        if (kShared) {
            landed(c);
            ldsm4t(uf, stage(c) + u1_off);
        }
        // ---- Y^T = S^T W^T for this warp's 16 tokens: even and odd k-steps in chains of their own
        float y[2][2][4] = {};
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
            uint32_t a[4];
            ldsm4(a, a_s + ks * 32);
            if (kShared) load_w(wf[0], stage(c), ks);
            const uint32_t(&w)[4] = wf[kShared ? 0 : ks];
#pragma unroll
            for (int n = 0; n < 2; ++n) mma_16816(y[ks & 1][n], a, w[2 * n], w[2 * n + 1]);
        }
        if (!kShared && more) {
            landed(c + 1);
            load_all_w(c + 1);
        }
        // ---- U^T = U1^T - Y^T
#pragma unroll
        for (int n = 0; n < 2; ++n)
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const uint32_t u1 = kRuns ? uf[2 * n + half] & u1_mask : uf[2 * n + half];
                const float lo = __uint_as_float(u1 << 16) - (y[0][n][2 * half] + y[1][n][2 * half]);
                const float hi = __uint_as_float(u1 & 0xFFFF0000u) - (y[0][n][2 * half + 1] + y[1][n][2 * half + 1]);
                *reinterpret_cast<uint32_t*>(u_s + (ge + 8 * half) * kScanLdU + wq * 16 + n * 8 + gk) = pack_bf16(lo, hi);
            }
        const float g = __shfl_sync(0xffffffffu, g_cur, c & 31);
        if ((c & 31) == 31) g_cur = c + 1 + lane < nchunk ? gc[c + 1 + lane] : 1.0f;
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
            for (int x = 0; x < 4; ++x) st[n][x] *= g;
        group_sync();
        // ---- S^T = g S^T + U^T Khat for this warp's 32 keys
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
            uint32_t a[4];
            ldsm4(a, a_u + ks * 32);
            if (kShared) {
                load_k(kf[0][0], stage(c), ks, 0);
                load_k(kf[0][1], stage(c), ks, 1);
            }
            const uint32_t(&kk)[2][4] = kf[kShared ? 0 : ks];
#pragma unroll
            for (int n = 0; n < 4; ++n) mma_16816(st[n], a, kk[n >> 1][(n & 1) * 2], kk[n >> 1][(n & 1) * 2 + 1]);
        }
        if (kShared) release(c);
        if (more) {
            if (!kShared) {
                load_all_k(c + 1);
                release(c + 1);   // chunk c + 1 is in registers
            }
            put_s();
            group_sync();
        }
    }
    if (dead) return;
    float* nrow = p.next + (srow - p.state);
    if (kRuns) nrow += (bh * (2 * p.runs - 2) + (run == 0 ? 0 : 2 * run - 1 + (is_m ? 1 : 0))) * (size_t)(kTile * kTile);
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int x = 0; x < 4; ++x) nrow[(size_t)(n * 8 + (x & 1)) * kTile + (x >> 1) * 8] = st[n][x];
}

// S and its bf16 copy <- the result of the walk, if no wait of any of its CTAs (or of the kernel before it)
// expired.  A head's slabs are walked by CTAs that know nothing of one another: were each to store its own
// columns of S, one that gives up after another has finished would leave the head half old, half new.  2.2 us
// behind the walk; commit_tokens of 12 heads x 4680 tokens 90.2 -> 91.7.
constexpr int kPublishThreads = 256;   // four values each
__global__ void __launch_bounds__(kPublishThreads) tc_token_publish_kernel(const TcTokenParams p)
{
    const size_t i = ((size_t)blockIdx.x * kPublishThreads + threadIdx.x) * 4;
    grid_dependency_sync();
    const uint32_t err = p.status[kStatusError];
    const float4 v = *reinterpret_cast<const float4*>(p.next + i);   // (on its way beside the status word)
    if (err != 0u) return;
    *reinterpret_cast<float4*>(p.state + i) = v;
    *reinterpret_cast<uint2*>(p.state_bf16 + i) = make_uint2(pack_bf16(v.x, v.y), pack_bf16(v.z, v.w));
}

// The same behind a walk in runs: S <- M_r S + N_r for r = 1 .. runs - 1, from the first run's S.  One CTA per
// kJoinCols value columns of a head (columns do not mix), in fp32 FMAs: the state is not rounded between chunks, and
// is not here.  A thread has 2 columns of 4 rows.  The kernel is one round of loads (72 KB per CTA) and 1.3 us of
// multiplications; M of the next run is on its way while this one is used.
constexpr int kJoinCols = 16, kJoinThreads = 256;
constexpr int kJoinLdM = kTile + 4;   // fp32 row stride: the four rows a warp reads at a time lie in different banks
constexpr int kJoinMatBytes = kTile * kJoinLdM * 4;
constexpr int join_smem_bytes(int runs) { return (runs > 2 ? 2 : 1) * kJoinMatBytes + kTile * kJoinCols * 4; }
__global__ void __launch_bounds__(kJoinThreads) tc_token_join_kernel(const TcTokenParams p)
{
    extern __shared__ __align__(16) float join_smem[];
    float* Ss = join_smem + (p.runs > 2 ? 2 : 1) * kTile * kJoinLdM;
    const int tid = threadIdx.x;
    const size_t bh = blockIdx.x / (kTile / kJoinCols);
    const int e0 = (int)(blockIdx.x % (kTile / kJoinCols)) * kJoinCols;
    const int c2 = (tid & 7) * 2, r0 = tid >> 3;   // columns c2, c2 + 1 of rows r0 + 32 i
    const float* base = p.next + bh * (2 * p.runs - 1) * (size_t)(kTile * kTile);
    grid_dependency_sync();
    const uint32_t err = p.status[kStatusError];
    auto fetch_m = [&](int r) {
        const float* M = base + (size_t)(2 * r) * kTile * kTile;
        const uint32_t dst = smem_u32(join_smem + ((r - 1) & 1) * kTile * kJoinLdM);
#pragma unroll
        for (int i = 0; i < kTile * kTile / 4 / kJoinThreads; ++i) {
            const int c = tid + i * kJoinThreads;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + (uint32_t)((c >> 5) * kJoinLdM + (c & 31) * 4) * 4), "l"(M + c * 4)
                         : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    fetch_m(1);
    float2 S[4], out[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) S[i] = *reinterpret_cast<const float2*>(base + (size_t)(r0 + 32 * i) * kTile + e0 + c2);
    for (int r = 1; r < p.runs; ++r) {
        const float* N = base + (size_t)(2 * r - 1) * kTile * kTile;
#pragma unroll
        for (int i = 0; i < 4; ++i) out[i] = *reinterpret_cast<const float2*>(N + (size_t)(r0 + 32 * i) * kTile + e0 + c2);
        if (r > 1) __syncthreads();   // S and the other buffer of the run before have been read
        if (r + 1 < p.runs) fetch_m(r + 1);
#pragma unroll
        for (int i = 0; i < 4; ++i) *reinterpret_cast<float2*>(Ss + (r0 + 32 * i) * kJoinCols + c2) = S[i];
        if (r + 1 < p.runs) asm volatile("cp.async.wait_group 1;" ::: "memory");
        else asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        const float* Ms = join_smem + ((r - 1) & 1) * kTile * kJoinLdM;
#pragma unroll 4
        for (int q = 0; q < kTile; q += 4) {
            float2 s[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) s[x] = *reinterpret_cast<const float2*>(Ss + (q + x) * kJoinCols + c2);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 m = *reinterpret_cast<const float4*>(Ms + (r0 + 32 * i) * kJoinLdM + q);
                out[i].x = fmaf(m.x, s[0].x, out[i].x); out[i].y = fmaf(m.x, s[0].y, out[i].y);
                out[i].x = fmaf(m.y, s[1].x, out[i].x); out[i].y = fmaf(m.y, s[1].y, out[i].y);
                out[i].x = fmaf(m.z, s[2].x, out[i].x); out[i].y = fmaf(m.z, s[2].y, out[i].y);
                out[i].x = fmaf(m.w, s[3].x, out[i].x); out[i].y = fmaf(m.w, s[3].y, out[i].y);
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) S[i] = out[i];
    }
    if (err != 0u) return;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const size_t at = (bh * kTile + r0 + 32 * i) * kTile + e0 + c2;
        *reinterpret_cast<float2*>(p.state + at) = S[i];
        *reinterpret_cast<uint32_t*>(p.state_bf16 + at) = pack_bf16(S[i].x, S[i].y);
    }
}

// The rotation table in the form the step kernel reads: half2 (cos, sin) per pair, 16 vectors of

// 4 pairs per token, stored so that the 32 tokens a warp owns are interleaved -- vector c of
// token l sits at uint4 index ((l / 32) * 16 + c) * 32 + l % 32 -- and each of a warp's 16 loads is
// one contiguous 512-byte segment.  Tokens past L (padding up to a whole tile) read as zero.
// fp16 keeps 11 bits of the unit-range values.
__global__ void pack_rope_kernel(const float* __restrict__ cos_t, const float* __restrict__ sin_t,
                                 __half2* __restrict__ out, int L, size_t total)
{
    size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= total) return;
    const int l = (int)(t / 64), m = (int)(t % 64);
    const int c = m >> 2, w = m & 3;
    const size_t dst = ((((size_t)(l >> 5) * 16 + c) * 32 + (l & 31)) << 2) + w;
    out[dst] = l < L ? __floats2half2_rn(cos_t[t], sin_t[t]) : __floats2half2_rn(0.0f, 0.0f);
}

// k_rot = RoPE(k) for bf16 [B, L, H, 128] from the packed half2 table: 16 threads per row (8 elements, 4 rotation
// pairs, one 16-byte table vector each), kRopeRows rows per thread with all loads ahead of the first use.  The same table
// rotates Q inside the step kernel.  Bound by memory, and where it is short by its latencies.  (With one row per thread,
// 64-bit index divisions and the step kernel's first Q tiles requested 0.6 us later and rotated 1.2 us later: 40.2 us per
// pass of 12 heads x 1560 tokens against 38.8.  The two changes were not timed apart.)
constexpr int kRopeRows = 4;
__global__ void __launch_bounds__(256) tc_rope_k_kernel(const uint4* k, const uint4* rope_h,
                                                        uint4* __restrict__ out, uint32_t L, uint32_t H, uint32_t rows)
{
    const uint32_t c = threadIdx.x & 15;             // vector of the 128-element row
    const uint32_t row0 = blockIdx.x * (16 * kRopeRows) + (threadIdx.x >> 4);
    const uint4* tab[kRopeRows];
#pragma unroll
    for (int i = 0; i < kRopeRows; ++i) {
        const uint32_t l = (row0 + i * 16) / H % L;  // token
        tab[i] = rope_h + ((size_t)(l >> 5) * 16 + c) * 32 + (l & 31);
    }
    grid_dependency_sync();
    uint4 raw[kRopeRows], cs[kRopeRows];
#pragma unroll
    for (int i = 0; i < kRopeRows; ++i) {
        if (row0 + i * 16 < rows) {
            raw[i] = k[(size_t)(row0 + i * 16) * 16 + c];
            cs[i] = *tab[i];
        }
    }
#pragma unroll
    for (int i = 0; i < kRopeRows; ++i) {
        if (row0 + i * 16 >= rows) return;
        uint32_t w[4] = {raw[i].x, raw[i].y, raw[i].z, raw[i].w};
        const uint32_t h2[4] = {cs[i].x, cs[i].y, cs[i].z, cs[i].w};
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            float cc, ss;
            unpack_cs(h2[m], cc, ss);
            const float x0 = __uint_as_float(w[m] << 16);
            const float x1 = __uint_as_float(w[m] & 0xFFFF0000u);
            w[m] = pack_bf16(x0 * cc - x1 * ss, x0 * ss + x1 * cc);
        }
        out[(size_t)(row0 + i * 16) * 16 + c] = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// out[h][o][i] = w[h][i][o] (bf16), or the identity when w is null: the K-major B operand of
// U = Q W_phi (B[n][k] = W[k][n]).
__global__ void transpose_map_kernel(const __nv_bfloat16* __restrict__ w, __nv_bfloat16* __restrict__ out,
                                     int D, size_t total)
{
    size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= total) return;
    int i = (int)(t % D);
    int o = (int)((t / D) % D);
    size_t hh = t / ((size_t)D * D);
    __nv_bfloat16 v;
    if (w != nullptr) v = w[(hh * D + i) * D + o];
    else v = __float2bfloat16_rn(i == o ? 1.0f : 0.0f);
    out[t] = v;
}

// Combines the parts of the split items of a step launch: a warp takes kMergeRows consecutive query
// rows of one tile (the item is decoded once per warp), a lane four output channels of each.  With
// part q's reference maximum m_q, row sum l_q and unnormalised row O_q:
//   out = sum_q 2^(m_q - m) O_q / sum_q 2^(m_q - m) l_q,   m = max_q m_q,   summed in part order.
constexpr int kMergeRows = 4;
__global__ void __launch_bounds__(256)
tc_split_merge_kernel(const TcStepParams p)
{
    const int warp = (int)((blockIdx.x * 256u + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    constexpr int kWarpsPerTile = kTile / kMergeRows;
    const int r0 = (warp % kWarpsPerTile) * kMergeRows, t = (warp / kWarpsPerTile) & 1, slot = warp / (2 * kWarpsPerTile);
    const bool in_range = slot < p.n_items - p.n_whole;
    Item it;
    if (in_range) it = decode_item<false>(p.n_whole + slot, p);
    const int k = p.k_split;
    const size_t tp0 = ((size_t)slot * 2 + t) * k;
    grid_dependency_sync();   // the step kernel has finished, its writes are visible
    if (!in_range || t >= it.ntile || p.status[kStatusError] != 0u) return;
    const int row0 = it.row0[t] + r0;
    __nv_bfloat16* obase = p.out + (((size_t)it.b[t] * p.s.L + row0) * p.s.H + it.h[t]) * kTile + lane * 4;
    // all loads of the warp's rows go out before the first use
    float2 ml[kMergeRows][kMaxSplit];
    float4 x[kMergeRows][kMaxSplit];
#pragma unroll
    for (int i = 0; i < kMergeRows; ++i) {
#pragma unroll
        for (int q = 0; q < kMaxSplit; ++q) {
            if (q < k && row0 + i < p.s.L) {
                const size_t rr = (tp0 + q) * kTile + r0 + i;
                ml[i][q] = *reinterpret_cast<const float2*>(p.split_ml + rr * 2);
                x[i][q] = *reinterpret_cast<const float4*>(p.split_o + rr * kTile + lane * 4);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < kMergeRows; ++i) {
        if (row0 + i >= p.s.L) break;
        float m_all = -INFINITY;
#pragma unroll
        for (int q = 0; q < kMaxSplit; ++q)
            if (q < k) m_all = fmaxf(m_all, ml[i][q].x);
        float l_all = 0.0f;
        float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
        for (int q = 0; q < kMaxSplit; ++q) {
            if (q < k) {
                const float wq = ex2_approx(ml[i][q].x - m_all);
                l_all = fmaf(wq, ml[i][q].y, l_all);
                acc.x = fmaf(wq, x[i][q].x, acc.x);
                acc.y = fmaf(wq, x[i][q].y, acc.y);
                acc.z = fmaf(wq, x[i][q].z, acc.z);
                acc.w = fmaf(wq, x[i][q].w, acc.w);
            }
        }
        const float inv = 1.0f / l_all;
        *reinterpret_cast<uint2*>(obase + (size_t)i * p.s.H * kTile) =
            make_uint2(pack_bf16(acc.x * inv, acc.y * inv), pack_bf16(acc.z * inv, acc.w * inv));
    }
}

// The work items of a step launch and how its last wave is cut.
void plan_items(const StepArgs& a, int num_sms, TcStepParams& p)
{
    p.Lk = a.Lk > 0 ? a.Lk : a.s.L;
    p.n_q = (a.s.L + kTile - 1) / kTile;
    p.n_kv = (p.Lk + kTile - 1) / kTile;
    const int bh = a.s.B * a.s.H;
    p.n_pair_items = bh * (p.n_q / 2);
    p.n_items = p.n_pair_items + ((p.n_q & 1) ? (bh + 1) / 2 : 0);   // ragged tiles go two by two
    const bool elem_gate = a.gate_mode == 2 && a.gate != nullptr;
    // The last wave: `rem` items on num_sms SMs.  Cut into k key ranges, the wave takes
    // ceil(rem k / SMs) rounds of one part each; a part costs its share of the key iterations plus
    // what every item costs (the readout iteration, the hand-over between items) plus the exchange
    // of the partial rows -- measured: 3.3 k clk per iteration, 10.8 k per item, about 6 k for the
    // exchange.  Take the k that makes the wave shortest, if that is shorter than leaving it whole.
    // (At 3.7 k, what an iteration took before the issuers took turns, 26 to 28 key tiles were still cut in three
    // where a third costs more than it saves: 6 heads x 3300 tokens 68 us, whole 62; 29 x 3456 218, 204;
    // 17 x 3584 139, 125.)
    p.n_whole = p.n_items;
    p.k_split = 1;
    if (!elem_gate && a.split_o != nullptr) {
        const int waves = (p.n_items + num_sms - 1) / num_sms;
        const int rem = p.n_items - (waves - 1) * num_sms;
        const float iter = 3.31f, fixed = 10.8f, exchange = 6.0f;
        float best = (p.n_kv + 1) * iter + fixed;
        for (int k = 2; k <= kMaxSplit; ++k) {
            if (p.n_kv < 4 * k || (long)rem * k * 2 > a.split_tile_parts) break;
            const float part = ((float)p.n_kv / k + 1.0f) * iter + fixed + exchange;
            const float cost = (float)((rem * k + num_sms - 1) / num_sms) * part;
            if (cost < 0.95f * best) { best = cost; p.k_split = k; }
        }
        if (p.k_split > 1) p.n_whole = p.n_items - rem;
    }
    p.n_sched = p.n_whole + (p.n_items - p.n_whole) * p.k_split;
}

std::mutex g_setup_mutex;
DeviceSetup g_setup[kMaxDevices];

int device_setup(int* num_sms)
{
    return device_setup_once(g_setup_mutex, g_setup, [] {
        cudaError_t e = opt_in_smem(tc_step_kernel<false, false>, kSmemBytes);
        if (e == cudaSuccess) e = opt_in_smem(tc_step_kernel<true, false>, kSmemBytes);
        if (e == cudaSuccess) e = opt_in_smem(tc_step_kernel<false, true>, kSmemBytes);
        if (e == cudaSuccess) e = opt_in_smem(tc_token_prepare_kernel, kTPSmemBytes);
        if (e == cudaSuccess) e = opt_in_smem(tc_token_scan_kernel<1, false, false>, ScanCfg<1, false>::kSmemBytes);
        if (e == cudaSuccess) e = opt_in_smem(tc_token_scan_kernel<2, false, false>, ScanCfg<2, false>::kSmemBytes);
        if (e == cudaSuccess) e = opt_in_smem(tc_token_scan_kernel<1, false, true>, ScanCfg<1, false>::kSmemBytes);
        if (e == cudaSuccess) e = opt_in_smem(tc_token_scan_kernel<2, false, true>, ScanCfg<2, false>::kSmemBytes);
        if (e == cudaSuccess) e = opt_in_smem(tc_token_join_kernel, kMaxSmemPerCta);
        if (e == cudaSuccess) e = opt_in_smem(tc_token_scan_kernel<2, true, false>, ScanCfg<2, true>::kSmemBytes);
        return e;
    }, num_sms);
}

}  // namespace

bool tc_supported(const arl2_config& c)
{
    return c.io_dtype == ARL2_BF16 && c.D == kTile && !(c.flags & ARL2_FLAG_FORCE_SIMT);
}

int tc_prepare_map(const void* w, __nv_bfloat16* w_op, int H, cudaStream_t st)
{
    size_t total = (size_t)H * kTile * kTile;
    transpose_map_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(
        static_cast<const __nv_bfloat16*>(w), w_op, kTile, total);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) { set_error("launch of transpose_map_kernel failed: %s", cudaGetErrorString(e)); return ARL2_ERR_CUDA; }
    return 1;
}

int tc_rope_k(const Shape& s, const void* k, const void* rope_h, void* k_rot, cudaStream_t st)
{
    const size_t rows = (size_t)s.B * s.L * s.H;
    if (rows >= ((size_t)1 << 32) - 16 * kRopeRows) { set_error("tc_rope_k: too many rows"); return ARL2_ERR_UNSUPPORTED; }
    const cudaError_t e = launch_kernel(tc_rope_k_kernel, dim3((unsigned)((rows + 16 * kRopeRows - 1) / (16 * kRopeRows))), 256, 0, st,
                                        static_cast<const uint4*>(k), static_cast<const uint4*>(rope_h), static_cast<uint4*>(k_rot),
                                        (uint32_t)s.L, (uint32_t)s.H, (uint32_t)rows);
    if (e != cudaSuccess) { set_error("launch of tc_rope_k_kernel failed: %s", cudaGetErrorString(e)); return ARL2_ERR_CUDA; }
    return 1;
}

int tc_prepare_rope(const float* cos_t, const float* sin_t, void* out, int L, cudaStream_t st)
{
    size_t total = (size_t)((L + kTile - 1) / kTile) * kTile * (kTile / 2);   // padded to whole tiles
    pack_rope_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(cos_t, sin_t, static_cast<__half2*>(out), L,
                                                                         total);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) { set_error("launch of pack_rope_kernel failed: %s", cudaGetErrorString(e)); return ARL2_ERR_CUDA; }
    return 1;
}

int tc_step_ctas(const StepArgs& a, int* ctas, int* num_sms)
{
    if (int r = device_setup(num_sms)) return r;
    TcStepParams p;
    plan_items(a, *num_sms, p);
    *ctas = p.n_sched < *num_sms ? p.n_sched : *num_sms;
    return 0;
}

int tc_step(const StepArgs& a, const __nv_bfloat16* wq_op, const __nv_bfloat16* state_bf16, cudaStream_t st)
{
    int num_sms = 0;
    if (int r = device_setup(&num_sms)) return r;
    CUtensorMap tm_q, tm_k, tm_v, tm_w, tm_s, tm_o;
    if (int r = make_map_blhd(&tm_q, a.q, a.s)) return r;
    if (int r = make_map_blhd(&tm_o, a.out, a.s, 32)) return r;
    Shape ks = a.s;
    ks.L = a.Lk > 0 ? a.Lk : a.s.L;   // K and V may be a longer cache
    if (int r = make_map_blhd(&tm_k, a.k_rot, ks)) return r;
    if (int r = make_map_blhd(&tm_v, a.v, ks)) return r;
    if (int r = make_map_rows(&tm_w, wq_op, (size_t)a.s.H * kTile)) return r;
    if (int r = make_map_rows(&tm_s, state_bf16, (size_t)a.s.B * a.s.H * kTile)) return r;
    TcStepParams p;
    p.s = a.s;
    p.gate = a.gate;
    p.gate_mode = a.gate_mode;
    p.rope_cos = a.rope_cos;
    p.rope_sin = a.rope_sin;
    p.rope_h = static_cast<const uint4*>(a.rope_h);
    p.out = static_cast<__nv_bfloat16*>(a.out);
    p.status = a.status;
    p.spin_limit = a.wait_limit ? a.wait_limit - 1 : kSpinLimit;
    // two item counters alternate between launches: a launch uses one and clears the other
    p.sched_counter = a.status + kStatusSched + (a.launch_parity & 1);
    p.sched_next = a.status + kStatusSched + ((a.launch_parity + 1) & 1);
    const bool elem_gate = p.gate_mode == 2 && p.gate != nullptr;
    plan_items(a, num_sms, p);
    p.split_o = a.split_o;
    p.split_ml = a.split_ml;
    const int grid = p.n_sched < num_sms ? p.n_sched : num_sms;
    p.one_item = p.n_sched == grid ? 1 : 0;
    // After the kernel that makes K (the rotation, or the commit kernel of a clean pass) barriers, tensor memory, the first Q
    // tiles and their rotation run ahead of the wait; with K as the caller gave it the kernel before may be the one that
    // makes Q.  12 heads x 1560 tokens 44.1 -> 42.5 us per pass, 3 x 12 x 1001 38.8 -> 34.9, 2 heads x 300 22.5 -> 18.4.
    p.k_made_before = a.k_made_before ? 1 : 0;
    auto kernel = elem_gate ? tc_step_kernel<true, false> : p.k_split > 1 ? tc_step_kernel<false, true> : tc_step_kernel<false, false>;
    cudaError_t e = launch_kernel(kernel, dim3((unsigned)grid), kThreads, kSmemBytes, st, tm_q, tm_k, tm_v, tm_w, tm_s, tm_o, p);
    if (e != cudaSuccess) { set_error("launch of tc_step_kernel failed: %s", cudaGetErrorString(e)); return ARL2_ERR_CUDA; }
    if (p.k_split == 1) return 1;
    // the parts' rows are combined by a second, small kernel (one warp per row); it may start
    // before the step kernel ends and waits for it at its griddepcontrol.wait
    const long warps = (long)(p.n_items - p.n_whole) * 2 * (kTile / kMergeRows);
    e = launch_kernel(tc_split_merge_kernel, dim3((unsigned)((warps + 7) / 8)), 256, 0, st, p);
    if (e != cudaSuccess) { set_error("launch of tc_split_merge_kernel failed: %s", cudaGetErrorString(e)); return ARL2_ERR_CUDA; }
    return 2;
}

// What a chunk of the walk takes with one slab per SM and with two, and what runs cost on top (us; tc_token_join_kernel instead of
// tc_token_publish_kernel): fitted to whole calls of 2 to 12 heads x 300 to 4680 tokens, each with 1 to 4 runs.
// us per pass, one walk and with the runs this gives: 12 heads x 4680 tokens 83.3 -> 76.4 (2 runs, two slabs per SM),
// 5 x 4680 69.0 -> 52.0 (2), 2 x 4680 60.1 -> 39.3 (3), 2 x 3 x 2000 37.1 -> 31.9 (2).  Two runs where they are not taken: 12 x 1560
// 40.8 and 41.9, 8 x 1000 27.4 and 29.5, 2 x 600 23.6 and 24.5.
constexpr float kWalkChunk = 0.61f, kWalkChunk2 = 0.90f, kJoinFirst = 5.0f, kJoinMore = 4.0f;
constexpr int kMaxRuns = 4;

// Eq. 4 token by token with per-token gates on the tensor-core path (bf16 I/O, D = 128).  The
// scratch tensors of `a` (sized for the fp32 plain-FMA version) are used as bf16 here.
int tc_commit_tokens(const TokenCommitArgs& a, const __nv_bfloat16* wk_op, const __nv_bfloat16* wv_op,
                     const void* rope_h, uint32_t* status, cudaStream_t st)
{
    int num_sms = 0;
    if (int r = device_setup(&num_sms)) return r;
    if (a.state_bf16 == nullptr) { set_error("tc_commit_tokens: needs the bf16 copy of the state"); return ARL2_ERR_INVALID_ARG; }
    TcTokenParams p;
    p.s = a.s;
    p.rope_h = static_cast<const uint4*>(rope_h);
    p.alpha = a.alpha;
    p.beta = a.beta;
    p.w = reinterpret_cast<__nv_bfloat16*>(a.w);
    p.kh = reinterpret_cast<__nv_bfloat16*>(a.kh);
    p.u1 = reinterpret_cast<__nv_bfloat16*>(a.u1);
    p.gc = a.gc;
    p.state = a.state;
    p.state_bf16 = a.state_bf16;
    p.next = a.next;
    p.status = status;
    p.spin_limit = a.wait_limit ? a.wait_limit - 1 : kSpinLimit;
    p.walk_limit = a.walk_limit;
    p.ntile = (a.s.L + kTile - 1) / kTile;
    p.nchunk = (a.s.L + kTokC - 1) / kTokC;
    p.decayed = a.decayed ? 1 : 0;
    const size_t rows = (size_t)a.s.B * a.s.H * p.ntile * kTile;
    if (rows >= ((size_t)1 << 31)) { set_error("tc_commit_tokens: too many rows"); return ARL2_ERR_UNSUPPORTED; }
    // Value columns per scan CTA: 16 while that leaves one CTA per SM (the walk is a latency chain), 32
    // beyond (half the L2 traffic), two such CTAs per SM when even those do not fit beside one another (40 heads:
    // 157 -> 113 us for the walk; four slabs in one CTA took 205: its 16 warps load 139 KB of fragments per chunk).
    const long heads = (long)a.s.B * a.s.H;
    // Runs of chunks walked side by side, where that is shorter than one walk (tc_token_scan_kernel).  A run more is 16 slabs
    // per head more; the slabs have an SM each, or two share one, and the scratch has to hold 2 runs - 1 matrices per head.
    const auto walk_ctas = [&](int runs, int per) { return heads * 8 * (2 * runs - 1) / per; };
    p.runs = 1;
    float best = kWalkChunk * (float)p.nchunk;
    for (int r = 2; r <= kMaxRuns && walk_ctas(r, 2) <= num_sms && 2 * r - 1 <= a.next_slots; ++r) {
        const float chunk = walk_ctas(r, 1) <= num_sms ? kWalkChunk : kWalkChunk2;
        const float t = chunk * (float)((p.nchunk + r - 1) / r) + kJoinFirst + kJoinMore * (float)(r - 2);
        if (t < 0.97f * best) { best = t; p.runs = r; }
    }
    p.run_chunks = (p.nchunk + p.runs - 1) / p.runs;
    p.runs = (p.nchunk + p.run_chunks - 1) / p.run_chunks;   // (none is empty)
    const int slabs = walk_ctas(p.runs, 1) <= num_sms ? 1 : 2;
    const bool shared_sm = heads * 4 > num_sms;
    CUtensorMap tm_k, tm_v, tm_wk, tm_wv, tm_w, tm_kh, tm_u1;
    if (int r = make_map_blhd(&tm_k, a.k, a.s)) return r;
    if (int r = make_map_blhd(&tm_v, a.v, a.s)) return r;
    if (int r = make_map_rows(&tm_wk, wk_op, (size_t)a.s.H * kTile)) return r;
    if (int r = make_map_rows(&tm_wv, wv_op, (size_t)a.s.H * kTile)) return r;
    CUtensorMap out_w, out_u1;   // whole tiles, written by the prepare kernel
    if (int r = make_map_rows(&out_w, p.w, rows)) return r;
    if (int r = make_map_rows(&out_u1, p.u1, rows)) return r;
    if (int r = make_map_rows(&tm_w, p.w, rows, kTokC)) return r;
    if (int r = make_map_rows(&tm_kh, p.kh, rows, kTokC)) return r;
    if (int r = make_map_rows(&tm_u1, p.u1, rows, kTokC, slabs * kScanSlab, false)) return r;
    dim3 grid1(p.ntile, a.s.H, a.s.B);
    cudaError_t e = launch_kernel(tc_token_prepare_kernel, grid1, kTPThreads, kTPSmemBytes, st, tm_k, tm_v, tm_wk, tm_wv, out_w, out_u1, p);
    if (e != cudaSuccess) { set_error("launch of tc_token_prepare_kernel failed: %s", cudaGetErrorString(e)); return ARL2_ERR_CUDA; }
    dim3 grid2((2 * p.runs - 1) * (kTile / (slabs * kScanSlab)), a.s.H, a.s.B);
    if (p.runs > 1 && slabs == 1)
        e = launch_kernel(tc_token_scan_kernel<1, false, true>, grid2, ScanCfg<1, false>::kThreads, ScanCfg<1, false>::kSmemBytes, st, tm_w, tm_kh, tm_u1, p);
    else if (p.runs > 1)
        e = launch_kernel(tc_token_scan_kernel<2, false, true>, grid2, ScanCfg<2, false>::kThreads, ScanCfg<2, false>::kSmemBytes, st, tm_w, tm_kh, tm_u1, p);
    else if (slabs == 1)
        e = launch_kernel(tc_token_scan_kernel<1, false, false>, grid2, ScanCfg<1, false>::kThreads, ScanCfg<1, false>::kSmemBytes, st, tm_w, tm_kh, tm_u1, p);
    else if (!shared_sm)
        e = launch_kernel(tc_token_scan_kernel<2, false, false>, grid2, ScanCfg<2, false>::kThreads, ScanCfg<2, false>::kSmemBytes, st, tm_w, tm_kh, tm_u1, p);
    else
        e = launch_kernel(tc_token_scan_kernel<2, true, false>, grid2, ScanCfg<2, true>::kThreads, ScanCfg<2, true>::kSmemBytes, st, tm_w, tm_kh, tm_u1, p);
    if (e != cudaSuccess) { set_error("launch of tc_token_scan_kernel failed: %s", cudaGetErrorString(e)); return ARL2_ERR_CUDA; }
    if (p.runs > 1) {
        const int join_ctas = (int)heads * (kTile / kJoinCols);
        e = launch_kernel(tc_token_join_kernel, dim3((unsigned)join_ctas), kJoinThreads,
                          even_spread_smem(join_smem_bytes(p.runs), (join_ctas + num_sms - 1) / num_sms), st, p);
        if (e != cudaSuccess) { set_error("launch of tc_token_join_kernel failed: %s", cudaGetErrorString(e)); return ARL2_ERR_CUDA; }
        return 3;
    }
    e = launch_kernel(tc_token_publish_kernel, dim3((unsigned)(heads * (kTile * kTile / 4 / kPublishThreads))), kPublishThreads, 0, st, p);
    if (e != cudaSuccess) { set_error("launch of tc_token_publish_kernel failed: %s", cudaGetErrorString(e)); return ARL2_ERR_CUDA; }
    return 3;
}

}  // namespace arl2
