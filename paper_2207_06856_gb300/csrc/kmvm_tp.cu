// The tensor-core kernel MVM over pairs of row tiles (Eq. mvm; Sec. 4.1).
//
//   out_i = a^2 sum_j k(x_i, x_j) v_j (+ sigma^2 v_i)
//
// S = XA_i XB_j^T on the tensor cores with the norm terms folded into the
// contraction, the kernel function on the special function units, and an FP32
// accumulation of P V in TMEM:
//
//   O (rows i, columns r) += P (128 x 128) . Vt_j^T (128 x rv)   M = 128, N = rv, K = 128
//
// P never leaves TMEM: each epilogue thread reads its columns of a row of S and
// writes P as packed 16-bit pairs, which is the A operand (.ts form) of the value
// product.  Shared memory then carries only the operand tiles (X_j for S, Vt_j as
// the 128-byte-swizzled B operand), whose reads by the tensor core (4 KB + 4 KB per
// S instruction, 32 rv bytes per value-product instruction) stay far below its 128
// bytes per cycle.  With P in shared memory (written by the epilogue, read by the
// tensor core as a 256-row B operand) that port was 87 % busy and bound the kernel.
//
// The right-hand sides' hi and lo parts are 2 R of the rv = 16 ceil(2 R / 16)
// columns of N, so 17 right-hand sides cost N = 48.  With PSPLIT the kernel tile
// is carried as hi + lo (hi = k rounded to the operand format, lo = k - hi
// exactly before its own rounding).
//
// Work item = (pair of 128-row tiles, column split).  Warps: 0-15 epilogue
// (warpgroup q handles row tile q & 1: four warps per scheduler hide the TMEM
// latencies behind the special-function work), 16 TMA producer, then the MMA
// issuers, one or two per row tile.  The two row tiles share nothing but the
// operand stages, so one's barriers fall into the other's arithmetic.
//
// What paces the kernel besides the special-function rate is latency: a barrier
// probe or a tcgen05 operation of a warp beside four busy epilogue warps costs 100-300
// cycles.  So the epilogue tells the issuers by named barriers (a waiting warp takes
// no issue slots; as mbarriers polled by the issuers: 0.71 ms instead of 0.62 for the
// FP16 tile), each with one arrival per warp, and the run-time loops are not
// unrolled (unrolled, the kernel was 50 KB of code instead of 30 KB: 1.01 ms instead
// of 0.89 for the hi + lo tile).
//
// TMEM, one 512-column allocation per CTA.  WIDE (single-term P, R <= 32): per
// row tile S (128 columns), P (64) and O (64); S is released as soon as the
// epilogue has read it, so the next S and the value product run behind the
// epilogue's arithmetic.  Otherwise hi and lo of P fill exactly the columns of
// their S and overwrite it in place: a slot is 64 columns of a tile, and each row
// tile owns a ring of three 64-column buffers (two where O needs 128 columns, R > 32).
// With the FP32 value product (no P, no O) each row tile has two 128-column buffers.
//
// N = 65,536, d = 8, 17 columns, RBF, ms per launch (P in shared memory, one S and
// one value-product issuer -> this form): FP16 tile 0.774 -> 0.611, hi + lo tile and
// inputs 1.45 -> 0.867, of which 0.43 is the special-function time of one ex2 a pair.
// With HS (GP_MVM_HALF_EXP) the S product accumulates in FP16 and the
// epilogue evaluates 2^s in FP16 pairs.
//
// A single column split writes the output directly (scale, noise); several
// write their hi and lo sums to the partial buffer, which the split reduction
// adds up in a fixed order.  Every mbarrier wait is bounded; a wait that
// runs out records DEV_TIMEOUT, drains what was issued, frees TMEM and exits.
#include "gpk_internal.cuh"
#include "ptx.cuh"
#include "kfun.cuh"

namespace gpk {

namespace {

constexpr int kBM = 128;
constexpr int kBN = 128;
constexpr int kPairRows = 256;
constexpr int kMaxStages = 6;
constexpr int kEpiWarps = 16;
constexpr int kTmaWarp = kEpiWarps;
constexpr int kMmaWarp = kEpiWarps + 1;   // MMA issuers (row tile 0, 1; in place: S of both, then the value products
                                          // of both); the first owns the TMEM
constexpr int kMaxBufs = 6;               // S buffers: 2 x ring slot + row tile
constexpr uint32_t kTmemCols = 512;
constexpr int kMaxSmemBytes = 227 * 1024;   // opt-in maximum per CTA (512 B kept for static shared memory)
constexpr uint32_t kSpvVBytes = 128u * 4u * 4u;   // FP32 value product: 128 columns x 4 rows of FP32 v

struct TpSmem {
    uint32_t xbytes, stage_bytes;
    int stages;
    uint32_t total;   // dynamic shared memory to request (includes 1 KB alignment slack)
};

constexpr uint32_t kOneCtaSmem = 116u << 10;

__host__ __device__ inline TpSmem tp_smem(int k_pad, int rv) {
    TpSmem m;
    m.xbytes = (uint32_t)kBM * (uint32_t)k_pad * 2u;
    m.stage_bytes = m.xbytes + 2u * (uint32_t)rv * 128u;
    m.stages = 0;
    const uint32_t fixed = 1024u + 4u * m.xbytes;   // two buffers of the pair's row operands
    for (int s = kMaxStages; s >= 2; --s)
        if (fixed + (uint32_t)s * m.stage_bytes <= (uint32_t)kMaxSmemBytes - 512u) { m.stages = s; break; }
    m.total = fixed + (uint32_t)m.stages * m.stage_bytes;
    // More than half of the SM's shared memory: a CTA allocates all of TMEM, so a second one
    // on its SM (another stream's) would hold threads and registers only to wait for it.
    if (m.total < kOneCtaSmem) m.total = kOneCtaSmem;
    return m;
}

struct TpParams {
    int n_ip, n_jt, n_split, n_items;
    int k_pad, rv;        // rv: rows of Vt per tile (N of the value product)
    int lo_off;           // row of Vt (column of O) where the lo parts start; 0: no lo parts
    int stages;
    TpSmem sm;
    int nrhs;             // right-hand sides in use
    int spv;              // 1: FP32 value product; the V map is FP32, 128 columns x 4 rows per box
    int diag;             // square Matern-1/2 operator: P_ii = 0 on chip (exact diagonal added later)
    int64_t ld_part;      // n_ip * 256
    float* partial;       // [n_split][hi, lo][nrhs][ld_part]; FP32 value product: [n_split][column half][nrhs][ld_part]
    // direct output (n_split = 1): out[c][i] = outscale[c] O + noise Vnoise[c][i]
    float* out;
    int64_t ld_out, Nr, ld_v;
    const float* outscale;
    const float* Vnoise;
    float noise;
    const uint32_t* mask; // tile skipping: bit jt of word ip * mask_words + jt / 32 set = evaluate, or null
    int mask_words;
    int* err;
    uint64_t limit_ns;
};

struct TpBarriers {
    uint64_t full[kMaxStages];
    uint64_t empty[kMaxStages];
    // S and P buffers, [2 x ring slot + row tile]
    uint64_t s_full[kMaxBufs];
    uint64_t p_empty[kMaxBufs]; // P consumed by its value product (and, in place, S may be rewritten);
                                // FP32 value product: S read by the row tile's epilogue warps
    uint64_t o_full[2];         // per row tile, once per item with an evaluated tile
    uint64_t xi_full[2];
    uint64_t xi_empty[2];
    uint64_t drain[4];          // per issuing warp
};

// Named barriers between the 8 epilogue warps of a row tile (arrive) and its
// issuer (sync): S read into registers, P stored.  id 0 is __syncthreads.
constexpr uint32_t kBarThreads = 9 * 32;
constexpr uint32_t bar_s_read(uint32_t w) { return 1u + w; }        // WIDE: row tile
constexpr uint32_t bar_p_full(uint32_t buf) { return 3u + buf; }    // 2 x ring slot + row tile < 6

// WIDE (P beside S), in place (P over S, NG buffers per row tile), or FP32 value product.
enum TpMode { kWide = 0, kInPlace = 1, kSpv = 2 };
__host__ __device__ constexpr int tp_threads(int mode) { return (kEpiWarps + (mode == kInPlace ? 5 : 3)) * 32; }

// TMEM columns.
template <int MODE, int NG>
struct TpTmem {
    static constexpr uint32_t kS = MODE == kInPlace ? 64u : 128u;          // width of an S buffer
    static constexpr uint32_t s(uint32_t b, uint32_t w) { return (2u * b + w) * kS; }
    static constexpr uint32_t p(uint32_t b, uint32_t w) { return MODE == kWide ? 256u + w * 64u : s(b, w); }
    static constexpr uint32_t o(uint32_t w) { return MODE == kWide ? 384u + w * 64u : 128u * NG + w * (256u - 64u * NG); }
};

__device__ __forceinline__ void record_error(int* err, int code) { atomicCAS(err, 0, code); }

__device__ __forceinline__ void item_range(const TpParams& p, int item, int& ip, int& sp, int& j0, int& j1) {
    // 32-bit: n_split <= 16 and n_jt <= 2^24
    const uint32_t q = (uint32_t)item / (uint32_t)p.n_ip;
    sp = (int)q;
    ip = item - sp * p.n_ip;
    j0 = (int)(q * (uint32_t)p.n_jt / (uint32_t)p.n_split);
    j1 = (int)((q + 1u) * (uint32_t)p.n_jt / (uint32_t)p.n_split);
}

// Tile skipping (SKIP; compact support): a cleared bit of the mask means every kernel value of
// (row-tile pair ip, column tile jt) rounds to zero. Every role goes through the mask for itself, a
// word of 32 tiles at a time; the issuers and the epilogues take the stages as they come and need
// the number of tiles alone (but for Matern-1/2's diagonal). Tile by tile, in one kernel for both
// cases: 0.260 ms a launch for 16 far-apart clusters (N = 65,536, d = 8, 17 columns, 1 tile in 16
// evaluated) and, for 64 clusters, d = 3, 336 us a call at N = 65,536 and 992 at 131,072; like this
// 0.116 ms, 170 and 318 us.

// Evaluated column tiles of pair ip in [j0, j1).
template <int SKIP>
__device__ __forceinline__ int tile_count(const TpParams& p, int ip, int j0, int j1) {
    if constexpr (!SKIP) return j1 - j0;
    const uint32_t* m = p.mask + (int64_t)ip * p.mask_words;
    int n = 0;
#pragma unroll 1
    for (int w = j0 >> 5; 32 * w < j1; ++w) {
        uint32_t bits = __ldg(m + w);
        if (32 * w < j0) bits &= 0xffffffffu << (j0 - 32 * w);
        if (32 * w + 32 > j1) bits &= 0xffffffffu >> (32 * w + 32 - j1);
        n += __popc(bits);
    }
    return n;
}
// The first evaluated column tile of pair ip in [jt, j1), or j1.
template <int SKIP>
__device__ __forceinline__ int next_tile(const TpParams& p, int ip, int jt, int j1) {
    if constexpr (!SKIP) return jt;
    if (jt >= j1) return j1;
    const uint32_t* m = p.mask + (int64_t)ip * p.mask_words;
    int w = jt >> 5;
    uint32_t bits = __ldg(m + w) & (0xffffffffu << (jt & 31));
#pragma unroll 1
    while (bits == 0u) {
        if (32 * ++w >= j1) return j1;
        bits = __ldg(m + w);
    }
    jt = 32 * w + __ffs((int)bits) - 1;
    return jt < j1 ? jt : j1;
}

// ---- TMA producer (one thread) ------------------------------------------------
template <int SKIP>
__device__ void tp_producer(const TpParams& p, const CUtensorMap* tmA, const CUtensorMap* tmB,
                            const CUtensorMap* tmV, TpBarriers& bars, uint8_t* sSt, uint8_t* sXi, uint32_t xbytes,
                            uint32_t vtbytes) {
    uint32_t fills = 0, xi_loads = 0;
    bool ok = true;
    int ic = 0;
    const uint32_t S = (uint32_t)p.stages;
    const uint32_t kblk = (uint32_t)p.rv * 128u;
#pragma unroll 1
    for (int item = blockIdx.x; item < p.n_items; item += gridDim.x, ++ic) {
        int ip, sp, j0, j1;
        item_range(p, item, ip, sp, j0, j1);
        const int xb = ic & 1, use = ic >> 1;   // earlier uses of this buffer
        if (use >= 1 && !ptx::mbar_wait(&bars.xi_empty[xb], (use - 1) & 1, p.limit_ns)) { ok = false; break; }
        uint8_t* sX = sXi + (uint32_t)xb * 2u * xbytes;
        ptx::mbar_arrive_expect_tx(&bars.xi_full[xb], 2u * xbytes);
        ptx::tma_load_2d(sX, tmA, &bars.xi_full[xb], 0, ip * kPairRows);
        ptx::tma_load_2d(sX + xbytes, tmA, &bars.xi_full[xb], 0, ip * kPairRows + kBM);
        ++xi_loads;
#pragma unroll 1
        for (int jt = next_tile<SKIP>(p, ip, j0, j1); jt < j1; jt = next_tile<SKIP>(p, ip, jt + 1, j1)) {
            const uint32_t st = fills % S, u = fills / S;
            if (u > 0 && !ptx::mbar_wait_sleep(&bars.empty[st], (u - 1) & 1, p.limit_ns)) { ok = false; break; }
            uint8_t* sx = sSt + st * (xbytes + vtbytes);
            ptx::mbar_arrive_expect_tx(&bars.full[st], xbytes + (p.spv ? kSpvVBytes : vtbytes));
            ptx::tma_load_2d(sx, tmB, &bars.full[st], 0, jt * kBN);
            if (p.spv) {
                ptx::tma_load_2d(sx + xbytes, tmV, &bars.full[st], jt * kBN, 0);
            } else {
                ptx::tma_load_2d(sx + xbytes, tmV, &bars.full[st], jt * kBN, 0);
                ptx::tma_load_2d(sx + xbytes + kblk, tmV, &bars.full[st], jt * kBN + 64, 0);
            }
            ++fills;
        }
        if (!ok) break;
    }
    if (!ok) {
        record_error(p.err, DEV_TIMEOUT);
        // Let every copy this thread issued land before the CTA can exit.
        const uint32_t first = fills > S ? fills - S : 0;
#pragma unroll 1
        for (uint32_t f = first; f < fills; ++f) ptx::mbar_wait(&bars.full[f % S], (f / S) & 1, p.limit_ns);
#pragma unroll 1
        for (uint32_t q = xi_loads > 2 ? xi_loads - 2 : 0; q < xi_loads; ++q)
            ptx::mbar_wait(&bars.xi_full[q & 1], (q >> 1) & 1, p.limit_ns);
    }
}

// ---- MMA issuers (two converged warps, one per row tile) -----------------------------
// An issuer waits for the epilogue on named barriers: a waiting warp takes no issue
// slots, where a warp polling an mbarrier takes them, and queue entries of the unit
// the special-function instructions go through, from the epilogue warps beside it.
// The mbarriers it looks at (operand stage landed, P consumed) have normally
// completed before.  Every decision is warp-uniform; each tcgen05.mma and commit is
// issued by one elected lane.  The tensor pipe executes what the two warps issue in
// arrival order; their accumulators are disjoint TMEM columns.
//
// A bounded wait that runs out makes the role go on without further waits or tensor
// work: it still meets its named barriers, so that every warp reaches the end.
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, uint64_t limit_ns) {
    return __all_sync(0xffffffffu, ptx::mbar_wait(bar, parity, limit_ns));
}

// Walks the column tiles whose S is issued; runs one tile ahead of the value
// product, across items.
template <int MODE, int NG, int SKIP>
struct TpSIssue {
    using T = TpTmem<MODE, NG>;
    const TpParams& p;
    TpBarriers& bars;
    uint32_t aSt, aXi0, xbytes, stage_bytes, arow, hi_x, tmem, id, w, s_full;
    int item, xb = 0;
    int left = 0;               // evaluated tiles of the item still to be selected
    uint32_t ic = 0;            // items entered
    uint32_t st = 0, ph = 0;    // stage ring slot and its fill parity
    uint32_t b = 0, bph = 1;    // buffer ring slot; parity of its last release (first round: passes at once)
    bool have = true;           // a tile is selected (its stage has landed)
    bool ok = true;

    __device__ TpSIssue(const TpParams& p_, TpBarriers& bars_, const uint8_t* sSt, const uint8_t* sXi, uint32_t xbytes_,
                        uint32_t stage_bytes_, uint32_t tmem_, uint32_t id_, uint32_t w_)
        : p(p_), bars(bars_), xbytes(xbytes_), stage_bytes(stage_bytes_), tmem(tmem_), id(id_), w(w_) {
        aSt = ptx::smem_u32(sSt);
        aXi0 = ptx::smem_u32(sXi) + w * xbytes;
        arow = (uint32_t)p.k_pad * 2u;   // 32, 64 or 128 bytes
        hi_x = ptx::smem_desc_hi(8u * arow, (arow == 32) ? 6u : (arow == 64 ? 4u : 2u));
        s_full = ptx::smem_u32(&bars.s_full[w]);
        item = (int)blockIdx.x - (int)gridDim.x;
    }
    // Select the next evaluated tile; have = false after the last.
    __device__ __forceinline__ void next() {
#pragma unroll 1
        while (have) {
            if (left > 0) {
                --left;
                ok = ok && warp_wait(&bars.full[st], ph, p.limit_ns);
                return;
            }
            if (ic > 0 && ok) ptx::mma_commit_elect(&bars.xi_empty[xb]);   // the row tile's last use in its item
            item += (int)gridDim.x;
            if (item >= p.n_items) { have = false; return; }
            int ip, sp, j0, j1;
            item_range(p, item, ip, sp, j0, j1);
            left = tile_count<SKIP>(p, ip, j0, j1);
            xb = (int)(ic & 1u);
            ok = ok && warp_wait(&bars.xi_full[xb], (ic >> 1) & 1u, p.limit_ns);
            ++ic;
        }
    }
    // S of columns [h kS, (h + 1) kS) of the selected tile into the ring's next buffer.
    __device__ __forceinline__ void issue(uint32_t h) {
        if (ok) {
            const uint32_t la = ptx::smem_desc_lo(aXi0 + (uint32_t)xb * 2u * xbytes);
            const uint32_t lb = ptx::smem_desc_lo(aSt + st * stage_bytes + h * T::kS * arow);
            const uint32_t tD = tmem + T::s(b, w), bar = s_full + 16u * b;
            ptx::tc_fence_after();
            if (arow == 32u) ptx::mma_f16_ss_elect_commit<1>(tD, la, lb, hi_x, id, bar);
            else if (arow == 64u) ptx::mma_f16_ss_elect_commit<2>(tD, la, lb, hi_x, id, bar);
            else ptx::mma_f16_ss_elect_commit<4>(tD, la, lb, hi_x, id, bar);
        }
        if (++b == NG) { b = 0; bph ^= 1u; }
    }
    __device__ __forceinline__ void next_stage() {
        if (++st == (uint32_t)p.stages) { st = 0; ph ^= 1u; }
    }
};

// The value product of one slot, O (+)= P Vt^T over 128 (WIDE) or 64 columns, and
// its commit on `bar`.  lV: descriptor word of Vt, kb: 64-column K-block in 16-byte units.
template <int MODE, int PSPLIT>
__device__ __forceinline__ void tp_value_product(uint32_t tO, uint32_t tP, uint32_t lV, uint32_t kb, uint32_t id_pv,
                                                 uint32_t acc, uint32_t bar) {
    const uint32_t hi = ptx::smem_desc_hi(1024u, 2u);
    ptx::tc_fence_after();
    if constexpr (MODE == kWide) {
        ptx::mma_f16_ts4_elect<8, 16, 24>(tO, tP, lV, hi, id_pv, acc, 0u);
        ptx::mma_f16_ts4_elect<8, 16, 24>(tO, tP + 32u, lV + kb, hi, id_pv, 1u, bar);
    } else if constexpr (PSPLIT) {
        ptx::mma_f16_ts4_elect<8, 32, 40>(tO, tP, lV, hi, id_pv, acc, 0u);
        ptx::mma_f16_ts4_elect<8, 32, 40>(tO, tP + 16u, lV, hi, id_pv, 1u, bar);
    } else {
        ptx::mma_f16_ts4_elect<8, 32, 40>(tO, tP, lV, hi, id_pv, acc, bar);
    }
}

// WIDE, issuer of row tile w: S(t + 1) once the epilogue holds S(t) in registers,
// then O += P(t) Vt^T once it has stored P(t).  In place, value-product issuer
// (the S issuer of tp_issuer_s refills the buffers): O += P(q) Vt^T for each slot.
template <int MODE, int NG, int PSPLIT, int SKIP>
__device__ void tp_issuer(const TpParams& p, TpBarriers& bars, const uint8_t* sSt, const uint8_t* sXi, uint32_t xbytes,
                          uint32_t stage_bytes, uint32_t tmem, uint32_t id_s, uint32_t id_pv, uint32_t w) {
    using T = TpTmem<MODE, NG>;
    TpSIssue<MODE, NG, SKIP> si(p, bars, sSt, sXi, xbytes, stage_bytes, tmem, id_s, w);
    const uint32_t lV0 = ptx::smem_desc_lo(ptx::smem_u32(sSt) + xbytes), kb = (uint32_t)p.rv * 8u;
    const uint32_t p_empty = ptx::smem_u32(&bars.p_empty[w]);
    const uint32_t tO = tmem + T::o(w);
    uint32_t st = 0, ph = 0, b = 0;
    if constexpr (MODE == kWide) {
        si.next();
        if (si.have) { si.issue(0); si.next_stage(); }
    }
#pragma unroll 1
    for (int item = blockIdx.x; item < p.n_items; item += gridDim.x) {
        int ip, sp, j0, j1;
        item_range(p, item, ip, sp, j0, j1);
        uint32_t acc = 0;   // 0 for the item's first product (the epilogue has read O of the last item before
                            // it stores this item's first P)
#pragma unroll 1
        for (int n = tile_count<SKIP>(p, ip, j0, j1); n > 0; --n) {
            const uint32_t lV = lV0 + st * (stage_bytes >> 4);
            if constexpr (MODE == kWide) {
                // (this tile's stage landed before its S was issued)
                ptx::bar_sync(bar_s_read(w), kBarThreads);
                si.next();
                if (si.have) { si.issue(0); si.next_stage(); }
                ptx::bar_sync(bar_p_full(w), kBarThreads);
                if (si.ok) tp_value_product<MODE, PSPLIT>(tO, tmem + T::p(0, w), lV, kb, id_pv, acc, p_empty);
            } else {
                si.ok = si.ok && warp_wait(&bars.full[st], ph, p.limit_ns);
#pragma unroll
                for (uint32_t h = 0; h < 2; ++h) {
                    ptx::bar_sync(bar_p_full(2u * b + w), kBarThreads);
                    if (si.ok)
                        tp_value_product<MODE, PSPLIT>(tO, tmem + T::p(b, w), lV + h * kb, kb, id_pv, h > 0 ? 1u : acc,
                                                       p_empty + 16u * b);
                    if (++b == NG) b = 0;
                }
            }
            if (si.ok) ptx::mma_commit_elect(&bars.empty[st]);   // this row tile is done with X_j and Vt_j of the stage
            if (++st == (uint32_t)p.stages) { st = 0; ph ^= 1u; }
            acc = 1;
        }
        // An item without an evaluated tile has no O.  One with tiles meets the epilogue at
        // bar_p_full, after the epilogue's wait for the last such item's O: the issuer is
        // never two phases of o_full ahead, where the wait's parity would repeat.
        if (acc && si.ok) ptx::mma_commit_elect(&bars.o_full[w]);
    }
    const uint32_t dr = MODE == kInPlace ? 2u + w : w;
    ptx::mma_commit_elect(&bars.drain[dr]);
    warp_wait(&bars.drain[dr], 0, p.limit_ns);
    if (!si.ok && (threadIdx.x & 31) == 0) record_error(p.err, DEV_TIMEOUT);
}

// In place, S issuer of row tile w: S of each slot (64 columns of a tile) once the
// value product of the slot NG before it in the ring has completed.
template <int NG, int SKIP>
__device__ void tp_issuer_s(const TpParams& p, TpBarriers& bars, const uint8_t* sSt, const uint8_t* sXi,
                            uint32_t xbytes, uint32_t stage_bytes, uint32_t tmem, uint32_t id_s, uint32_t w) {
    TpSIssue<kInPlace, NG, SKIP> si(p, bars, sSt, sXi, xbytes, stage_bytes, tmem, id_s, w);
#pragma unroll 1
    for (si.next(); si.have && si.ok; si.next()) {
#pragma unroll
        for (uint32_t h = 0; h < 2; ++h) {
            si.ok = si.ok && warp_wait(&bars.p_empty[2u * si.b + w], si.bph, p.limit_ns);
            si.issue(h);
        }
        si.next_stage();
    }
    ptx::mma_commit_elect(&bars.drain[w]);
    warp_wait(&bars.drain[w], 0, p.limit_ns);
    if (!si.ok && (threadIdx.x & 31) == 0) record_error(p.err, DEV_TIMEOUT);
}

// Issuer of row tile w for the FP32 value product: S only, two buffers, each refilled once the
// row tile's epilogue warps have read it (p_empty, one arrival per warp). Here the waits are
// mbarriers with the suspend-time hint on both sides: this epilogue is bound by issue slots and
// registers, and one named barrier more in its loop spilled. N = 65,536, d = 8, hi + lo inputs, RBF, us
// a call for 1, 2 and 4 columns: named barrier 795 / 1,203 / 2,171, this form 769 / 1,137 / 2,077.
template <int NG, int SKIP>
__device__ void tp_issuer_spv(const TpParams& p, TpBarriers& bars, const uint8_t* sSt, const uint8_t* sXi,
                              uint32_t xbytes, uint32_t stage_bytes, uint32_t tmem, uint32_t id_s, uint32_t w) {
    TpSIssue<kSpv, NG, SKIP> si(p, bars, sSt, sXi, xbytes, stage_bytes, tmem, id_s, w);
    for (si.next(); si.have; si.next()) {
        si.ok = si.ok &&
                __all_sync(0xffffffffu, ptx::mbar_wait_sleep(&bars.p_empty[2u * si.b + w], si.bph, p.limit_ns));
        si.issue(0);
        si.next_stage();
    }
    ptx::mma_commit_elect(&bars.drain[w]);
    warp_wait(&bars.drain[w], 0, p.limit_ns);
    if (!si.ok && (threadIdx.x & 31) == 0) record_error(p.err, DEV_TIMEOUT);
}

template <int BF16>
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    if constexpr (BF16) {
        __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
        return *reinterpret_cast<uint32_t*>(&h);
    } else {
        __half2 h = __floats2half2_rn(lo, hi);
        return *reinterpret_cast<uint32_t*>(&h);
    }
}

// (l0, l1) = (k0, k1) minus the two halves of u, exact: one mixed-precision FMA each
// (1.004 -> 0.930 ms for the hi + lo MVM at N = 65,536, 17 columns, against unpacking
// to FP32 and subtracting).
template <int BF16>
__device__ __forceinline__ void sub_packed(float k0, float k1, uint32_t u, float& l0, float& l1) {
    if constexpr (BF16) {
        l0 = k0 - __uint_as_float(u << 16);
        l1 = k1 - __uint_as_float(u & 0xffff0000u);
    } else {
        asm("{\n\t.reg .b16 a, b, m;\n\t"
            "mov.b32 {a, b}, %2;\n\t"
            "mov.b16 m, 0xBC00;\n\t"   // -1
            "fma.rn.f32.f16 %0, a, m, %3;\n\t"
            "fma.rn.f32.f16 %1, b, m, %4;\n\t}"
            : "=f"(l0), "=f"(l1)
            : "r"(u), "f"(k0), "f"(k1));
    }
}

// Kernel values of 32 columns [col0, col0 + 32) of this thread's row, packed in
// pairs (and, with PSPLIT, split: pl holds the lo parts).
template <int KIND, int BF16, int PSPLIT>
__device__ __forceinline__ void tp_values(const uint32_t (&r)[32], int col0, int row, bool dtile, uint32_t (&pk)[16],
                                          uint32_t (&pl)[16]) {
#pragma unroll
    for (int e = 0; e < 16; ++e) {
        float k0 = kernel_from_s<KIND>(__uint_as_float(r[2 * e]));
        float k1 = kernel_from_s<KIND>(__uint_as_float(r[2 * e + 1]));
        if constexpr (KIND == GP_KERNEL_MATERN12) {
            if (dtile) {
                const int col = col0 + 2 * e;
                if (col == row) k0 = 0.0f;
                if (col + 1 == row) k1 = 0.0f;
            }
        }
        pk[e] = pack2<BF16>(k0, k1);
        if constexpr (PSPLIT) {
            float l0, l1;
            sub_packed<BF16>(k0, k1, pk[e], l0, l1);
            pl[e] = pack2<BF16>(l0, l1);
        }
    }
}

template <int KIND, int BF16, int PSPLIT, int HS, int MODE, int NG, int SKIP>
__device__ void tp_epilogue(const TpParams& p, TpBarriers& bars, uint32_t tmem, int wg, int wq, int lane) {
    using T = TpTmem<MODE, NG>;
    constexpr int H = kBN / (int)T::kS;
    const int tl = wg & 1, ch = wg >> 1;              // row tile of the pair, half of a slot's columns
    const uint32_t lane_off = (uint32_t)(wq * 32) << 16;
    const int row = wq * 32 + lane;                   // row within the tile
    uint32_t b = 0, ph = 0;                           // buffer ring slot and its fill parity
    uint32_t oph = 0;                                 // parity of the next O: items with an evaluated tile only
    bool ok = true;
#pragma unroll 1
    for (int item = blockIdx.x; item < p.n_items; item += gridDim.x) {
        int ip, sp, j0, j1;
        item_range(p, item, ip, sp, j0, j1);
        const int it = 2 * ip + tl;   // this warpgroup's row tile
        const int tiles = tile_count<SKIP>(p, ip, j0, j1);
#pragma unroll 1
        for (int n = tiles, jt = j0 - 1; n > 0; --n) {
            if constexpr (KIND == GP_KERNEL_MATERN12) jt = next_tile<SKIP>(p, ip, jt + 1, j1);   // (the diagonal)
            const bool dtile = (KIND == GP_KERNEL_MATERN12) && p.diag && (jt == it);
#pragma unroll
            for (int h = 0; h < H; ++h) {
                const uint32_t buf = 2u * b + (uint32_t)tl;
                ok = ok && warp_wait(&bars.s_full[buf], ph, p.limit_ns);
                ptx::tc_fence_after();
                const uint32_t tS = tmem + lane_off + T::s(b, (uint32_t)tl) + (uint32_t)ch * (T::kS / 2u);
                uint32_t pk[16], pl[16];
                if constexpr (MODE == kWide) {
                    const uint32_t tP = tmem + lane_off + T::p(b, (uint32_t)tl) + (uint32_t)ch * 32u;
                    uint32_t ra[32], rb[HS ? 1 : 32];
                    if constexpr (HS) {
                        // Half-precision kernel evaluation (RBF, FP16): the S tile comes from the
                        // MMA as FP16 (one rounding of the exp2 argument), is loaded packed in pairs,
                        // and 2^s is evaluated for both halves of a register by one ex2.approx.f16x2,
                        // whose output is already the packed FP16 P the value product reads: no
                        // FP32 -> FP16 conversion, one SFU instruction per two kernel values.
                        ptx::tmem_ld32_pack16(tS, ra);     // 64 FP16 columns in 32 registers
                        ptx::tmem_wait_ld();
                        ptx::tmem_reg_fence(ra);
                    } else {
                        ptx::tmem_ld32(tS, ra);
                        ptx::tmem_ld32(tS + 32u, rb);
                        ptx::tmem_wait_ld();
                        ptx::tmem_reg_fence(ra);
                        ptx::tmem_reg_fence(rb);
                    }
                    ptx::tc_fence_before();
                    ptx::bar_arrive(bar_s_read((uint32_t)tl), kBarThreads, ok);   // S is in registers
                    if constexpr (HS) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) pk[e] = ptx::ex2_h2(ra[e]);
                    } else {
                        tp_values<KIND, BF16, 0>(ra, ch * 64, row, dtile, pk, pl);
                    }
                    // P is free once the value product of the previous tile is done (first use: at once)
                    ok = ok && warp_wait(&bars.p_empty[buf], ph ^ 1u, p.limit_ns);
                    ptx::tc_fence_after();
                    ptx::tmem_st16(tP, pk);
                    if constexpr (HS) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) pk[e] = ptx::ex2_h2(ra[16 + e]);
                    } else {
                        tp_values<KIND, BF16, 0>(rb, ch * 64 + 32, row, dtile, pk, pl);
                    }
                    ptx::tmem_st16(tP + 16u, pk);
                } else {
                    // in place: hi over the first 16 of this thread's 32 columns of S, lo over the others
                    uint32_t ra[32];
                    if constexpr (HS) {
                        ptx::tmem_ld16_pack16(tS, pk);     // 32 FP16 columns in 16 registers
                        ptx::tmem_wait_ld();
                        ptx::tmem_reg_fence(pk);
#pragma unroll
                        for (int e = 0; e < 16; ++e) pk[e] = ptx::ex2_h2(pk[e]);
                    } else {
                        ptx::tmem_ld32(tS, ra);
                        ptx::tmem_wait_ld();
                        ptx::tmem_reg_fence(ra);
                        tp_values<KIND, BF16, PSPLIT>(ra, h * 64 + ch * 32, row, dtile, pk, pl);
                    }
                    ptx::tmem_st16(tS, pk);
                    if constexpr (PSPLIT) ptx::tmem_st16(tS + 16u, pl);
                }
                ptx::tmem_wait_st();
                ptx::tc_fence_before();
                ptx::bar_arrive(bar_p_full(buf), kBarThreads, ok);
                if (++b == NG) { b = 0; ph ^= 1u; }
            }
        }
        // O read-out: lanes are rows of the tile; this warpgroup's half of the right-hand sides.
        if (tiles > 0) {
            ok = ok && warp_wait(&bars.o_full[tl], oph, p.limit_ns);
            oph ^= 1u;
        }
        ptx::tc_fence_after();
        const int half = (p.nrhs + 1) >> 1;
        const int c0 = ch * half, c1 = ch ? p.nrhs : half;
        const uint32_t tO = tmem + lane_off + T::o((uint32_t)tl);
        const int64_t i = (int64_t)ip * kPairRows + tl * kBM + row;
#pragma unroll 1
        for (int c = c0; c < c1; c += 8) {   // warp-uniform
            uint32_t oh[8], ol[8];
            if (tiles > 0) {
                ptx::tmem_ld8(tO + (uint32_t)c, oh);
                ptx::tmem_ld8(tO + (uint32_t)(p.lo_off + c), ol);
                ptx::tmem_wait_ld();
                ptx::tmem_reg_fence(oh);
                ptx::tmem_reg_fence(ol);
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) oh[e] = ol[e] = 0u;   // every tile of the item was skipped
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int cc = c + e;
                if (cc < c1) {
                    const float hi = __uint_as_float(oh[e]), lo = __uint_as_float(ol[e]);
                    if (p.n_split > 1) {   // rows [split][hi, lo][column], summed in this order
                        const int parts = p.lo_off ? 2 : 1;
                        float* o = p.partial + ((int64_t)sp * parts * p.nrhs + cc) * p.ld_part + i;
                        *o = hi;
                        if (p.lo_off) o[(int64_t)p.nrhs * p.ld_part] = lo;
                    } else if (i < p.Nr) {
                        float v = (p.lo_off ? hi + lo : hi) * __ldg(p.outscale + cc);
                        if (p.noise != 0.0f) v = fmaf(p.noise, __ldg(p.Vnoise + (int64_t)cc * p.ld_v + i), v);
                        p.out[(int64_t)cc * p.ld_out + i] = v;
                    }
                }
            }
        }
        ptx::tc_fence_before();   // ordered before this item's successor by the next P's barrier
    }
    if (!ok) record_error(p.err, DEV_TIMEOUT);
}

// The FP32 value product (GP_MVM_FP32_PV, 1 to 4 right-hand sides): the
// epilogue keeps its kernel values in FP32 and forms sum_j k_ij v_j itself
// with FP32 FMAs, v_j read in FP32 from the stage (TMA box of 128 columns x 4
// rows; this warpgroup's 64 columns; broadcast 16-byte reads).  No P and no
// value-product MMAs: no rounding of the kernel values, and
// one column takes 769 us a call against 850 on the hi + lo tile (N = 65,536, d = 8, RBF;
// two 1,137 and four 2,077, where the hi + lo tile's time hardly changes).  Each warp releases
// the stage after its reads (16 arrivals), and writes its row sums of the item
// to the partial rows ch * R + r, which the split reduction adds up.
template <int KIND, int RN, int SKIP>
__device__ void tp_epilogue_spv(const TpParams& p, TpBarriers& bars, const uint8_t* sSt, uint32_t xbytes,
                                uint32_t vtbytes, uint32_t tmem, int wg, int wq, int lane) {
    const int tl = wg & 1, ch = wg >> 1;
    const uint32_t lane_off = (uint32_t)(wq * 32) << 16;
    const int row = wq * 32 + lane;
    const uint32_t S = (uint32_t)p.stages;
    const uint32_t stage_bytes = xbytes + vtbytes;
    uint32_t g = 0, st = 0, ph = 0;   // evaluated tiles; stage ring slot and its fill parity
    bool ok = true;
#pragma unroll 1
    for (int item = blockIdx.x; item < p.n_items; item += gridDim.x) {
        int ip, sp, j0, j1;
        item_range(p, item, ip, sp, j0, j1);
        const int it = 2 * ip + tl;
        float acc[RN];
#pragma unroll
        for (int r = 0; r < RN; ++r) acc[r] = 0.0f;
#pragma unroll 1
        for (int n = tile_count<SKIP>(p, ip, j0, j1), jt = j0 - 1; n > 0; --n) {
            if constexpr (KIND == GP_KERNEL_MATERN12) jt = next_tile<SKIP>(p, ip, jt + 1, j1);   // (the diagonal)
            const uint32_t buf = g & 1u;
            // hinted waits: a spinning warp would take the issue slots of the warps computing
            // beside it and of the S issuer on its scheduler (this epilogue is issue-bound)
            if (!__all_sync(0xffffffffu, ptx::mbar_wait_sleep(&bars.s_full[2 * buf + tl], (g >> 1) & 1, p.limit_ns) &&
                                             ptx::mbar_wait_sleep(&bars.full[st], ph, p.limit_ns))) {
                ok = false;
                break;
            }
            ptx::tc_fence_after();
            const uint32_t tS = tmem + lane_off + buf * 256u + (uint32_t)tl * 128u + (uint32_t)ch * 64u;
            const bool dtile = (KIND == GP_KERNEL_MATERN12) && p.diag && (jt == it);
            const float* vb = reinterpret_cast<const float*>(sSt + st * stage_bytes + xbytes) + ch * 64;
            // one 32-column half of S at a time (the register budget of 608 threads); the
            // buffer is released after the second load, while S of the next tile is
            // already being formed in the other one. From two columns on the halves are a loop
            // (two columns, as above: 1,169 us unrolled with 8 bytes of spills, 1,138 as a loop; one
            // column, Matern-3/2: 1,608 unrolled, 1,881 as a loop)
#pragma unroll(RN == 1 ? 2 : 1)
            for (int hh = 0; hh < 2; ++hh) {
                uint32_t rr[32];
                ptx::tmem_ld32(tS + 32u * (uint32_t)hh, rr);
                ptx::tmem_wait_ld();
                ptx::tmem_reg_fence(rr);
                if (hh == 1) {
                    ptx::tc_fence_before();
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(&bars.p_empty[2u * buf + (uint32_t)tl]);
                }
#pragma unroll
                for (int c4 = 0; c4 < 4; ++c4) {      // 16-byte chunk c: columns [8 c, 8 c + 8) of the 64
                    const int c = 4 * hh + c4;
                    float kv[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const int q = 8 * c + e;
                        float k = kernel_from_s<KIND>(__uint_as_float(rr[8 * c4 + e]));
                        if constexpr (KIND == GP_KERNEL_MATERN12) {
                            if (dtile && ch * 64 + q == row) k = 0.0f;
                        }
                        kv[e] = k;
                    }
#pragma unroll
                    for (int r = 0; r < RN; ++r) {
                        {
                            const float4 va = *reinterpret_cast<const float4*>(vb + r * 128 + 8 * c);
                            const float4 vc = *reinterpret_cast<const float4*>(vb + r * 128 + 8 * c + 4);
                            acc[r] = fmaf(kv[0], va.x, acc[r]);
                            acc[r] = fmaf(kv[1], va.y, acc[r]);
                            acc[r] = fmaf(kv[2], va.z, acc[r]);
                            acc[r] = fmaf(kv[3], va.w, acc[r]);
                            acc[r] = fmaf(kv[4], vc.x, acc[r]);
                            acc[r] = fmaf(kv[5], vc.y, acc[r]);
                            acc[r] = fmaf(kv[6], vc.z, acc[r]);
                            acc[r] = fmaf(kv[7], vc.w, acc[r]);
                        }
                    }
                }
            }
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&bars.empty[st]);   // this warp is done with the stage's Vt
            if (++st == S) { st = 0; ph ^= 1u; }
            ++g;
        }
        if (!ok) break;
#pragma unroll
        for (int r = 0; r < RN; ++r)   // RN = 1, 2 or 4 (3 runs as 4: the fourth row of v is zero)
            if (r < p.nrhs)
                p.partial[((int64_t)(2 * sp + ch) * p.nrhs + r) * p.ld_part + (int64_t)ip * kPairRows + tl * kBM + row] =
                    acc[r];
    }
    if (!ok) record_error(p.err, DEV_TIMEOUT);
}

// MODE and NG as in TpTmem (in place: NG = 3 when O takes 64 columns per row tile, 2 when it takes 128).
template <int KIND, int BF16, int PSPLIT, int HS, int SPV, int MODE, int NG, int SKIP>
__global__ void __launch_bounds__(tp_threads(MODE), 1)
kmvm_tp_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
               const __grid_constant__ CUtensorMap tmV, const TpParams p) {
    extern __shared__ uint8_t dsm[];
    __shared__ TpBarriers bars;
    __shared__ uint32_t tmem_slot;

    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(dsm) + 1023) & ~uintptr_t(1023));
    const TpSmem& m = p.sm;
    uint8_t* sSt = base;
    uint8_t* sXi = base + (uint32_t)p.stages * m.stage_bytes;

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // warp-uniform
    if (threadIdx.x == 0) {
#pragma unroll 1
        for (int b = 0; b < kMaxStages; ++b) {
            ptx::mbar_init(&bars.full[b], 1);
            ptx::mbar_init(&bars.empty[b], SPV ? kEpiWarps : 2);   // the two value products; FP32: each epilogue warp
        }
#pragma unroll 1
        for (int b = 0; b < kMaxBufs; ++b) {
            ptx::mbar_init(&bars.s_full[b], 1);
            ptx::mbar_init(&bars.p_empty[b], SPV ? kEpiWarps / 2 : 1);
        }
#pragma unroll 1
        for (int b = 0; b < 2; ++b) {
            ptx::mbar_init(&bars.xi_full[b], 1);
            ptx::mbar_init(&bars.xi_empty[b], 2);
            ptx::mbar_init(&bars.o_full[b], 1);
            ptx::mbar_init(&bars.drain[b], 1);
            ptx::mbar_init(&bars.drain[2 + b], 1);
        }
        ptx::fence_mbar_init();
    }
    if (warp == kTmaWarp && lane == 0) {
        ptx::tma_prefetch_desc(&tmA);
        ptx::tma_prefetch_desc(&tmB);
        ptx::tma_prefetch_desc(&tmV);
    }
    if (warp == kMmaWarp) ptx::tmem_alloc(&tmem_slot, kTmemCols);
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = tmem_slot;

    if (warp == kTmaWarp) {
        if (lane == 0) tp_producer<SKIP>(p, &tmA, &tmB, &tmV, bars, sSt, sXi, m.xbytes, m.stage_bytes - m.xbytes);
        __syncwarp();
    } else if (warp >= kMmaWarp) {
        constexpr int kW = (int)TpTmem<MODE, NG>::kS;
        const uint32_t id_s = HS ? ptx::idesc_f16_dh(kBM, kW) : ptx::idesc_f16(kBM, kW, BF16);
        const uint32_t w = (uint32_t)(warp - kMmaWarp) & 1u;
        if constexpr (MODE == kInPlace) {
            if (warp < kMmaWarp + 2)
                tp_issuer_s<NG, SKIP>(p, bars, sSt, sXi, m.xbytes, m.stage_bytes, tmem, id_s, w);
            else
                tp_issuer<MODE, NG, PSPLIT, SKIP>(p, bars, sSt, sXi, m.xbytes, m.stage_bytes, tmem, id_s,
                                                  ptx::idesc_f16(kBM, p.rv, BF16), w);
        } else if constexpr (SPV > 0)
            tp_issuer_spv<NG, SKIP>(p, bars, sSt, sXi, m.xbytes, m.stage_bytes, tmem, id_s, w);
        else
            tp_issuer<MODE, NG, PSPLIT, SKIP>(p, bars, sSt, sXi, m.xbytes, m.stage_bytes, tmem, id_s,
                                              ptx::idesc_f16(kBM, p.rv, BF16), w);
    } else {
        if constexpr (SPV > 0)
            tp_epilogue_spv<KIND, SPV, SKIP>(p, bars, sSt, m.xbytes, m.stage_bytes - m.xbytes, tmem, warp >> 2,
                                             warp & 3, lane);
        else
            tp_epilogue<KIND, BF16, PSPLIT, HS, MODE, NG, SKIP>(p, bars, tmem, warp >> 2, warp & 3, lane);
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    if (warp == kMmaWarp) ptx::tmem_dealloc(tmem, kTmemCols);
}

template <int KIND, int BF16, int PSPLIT, int HS, int SPV, int MODE, int NG>
cudaError_t launch_tp_mode(const TcPlan& plan, const TpParams& prm, const CUtensorMap& a, const CUtensorMap& b,
                           const CUtensorMap& v, cudaStream_t s) {
    const TpSmem& m = prm.sm;
    auto kfn = prm.mask ? kmvm_tp_kernel<KIND, BF16, PSPLIT, HS, SPV, MODE, NG, 1>
                        : kmvm_tp_kernel<KIND, BF16, PSPLIT, HS, SPV, MODE, NG, 0>;
    cudaError_t e = allow_smem(kfn, kMaxSmemBytes - 512);
    if (e != cudaSuccess) return e;
    kfn<<<plan.grid, tp_threads(MODE), m.total, s>>>(a, b, v, prm);
    return cudaGetLastError();
}

template <int KIND, int BF16, int PSPLIT, int HS = 0, int SPV = 0>
cudaError_t launch_tp_typed(const TcPlan& plan, const TpParams& prm, const CUtensorMap& a, const CUtensorMap& b,
                            const CUtensorMap& v, cudaStream_t s) {
    if constexpr (SPV > 0) {
        return launch_tp_mode<KIND, BF16, PSPLIT, HS, SPV, kSpv, 2>(plan, prm, a, b, v, s);
    } else {
        if (prm.rv > 64) return launch_tp_mode<KIND, BF16, PSPLIT, HS, 0, kInPlace, 2>(plan, prm, a, b, v, s);
        if constexpr (PSPLIT) return launch_tp_mode<KIND, BF16, PSPLIT, HS, 0, kInPlace, 3>(plan, prm, a, b, v, s);
        else return launch_tp_mode<KIND, BF16, PSPLIT, HS, 0, kWide, 1>(plan, prm, a, b, v, s);
    }
}

}  // namespace

// The operand sets this engine takes (rp: right-hand sides padded to 16, hi and
// lo padded separately); the others run on the one-tile engine.  At k_pad = 64 the line at 64
// columns dates from when P took shared memory; three stages of 48 KB would fit beyond it now.
bool tp_supported(int k_pad, int R_pad, int vsplit) {
    const int rp = R_pad * (1 + vsplit);
    return k_pad <= 64 && rp <= (k_pad == 64 ? 64 : 128) && rp % 32 == 0;
}

int tp_rv(int R, int vsplit) { return ((R * (1 + vsplit) + 15) / 16) * 16; }

TcPlan tp_plan(const Ctx* ctx, int64_t Nr, int64_t Nc, int R, int k_pad, int vsplit) {
    TcPlan p;
    p.engine = 1;
    p.k_pad = k_pad;
    p.R_pad = ((R + 15) / 16) * 16;
    p.rv = tp_rv(R, vsplit);
    const int n_it = (int)((Nr + kBM - 1) / kBM);
    p.n_it = (n_it + 1) / 2;                  // pairs of row tiles
    p.n_jt = (int)((Nc + kBN - 1) / kBN);
    p.Nr_pad = (int64_t)p.n_it * kPairRows;
    p.Nc_pad = (int64_t)p.n_jt * kBN;
    const int G = ctx->num_sms > 0 ? ctx->num_sms : 1;
    // Column split minimising the busiest CTA's work (waves x tiles per item
    // plus about two tiles of per-item cost) plus the reduction of the splits' hi and
    // lo rows (counted for one split too, which writes its output itself).
    int best = 1;
    double best_cost = 1e300;
    const int max_split = p.n_jt < 16 ? p.n_jt : 16;
    for (int sp = 1; sp <= max_split; ++sp) {
        const int64_t items = (int64_t)p.n_it * sp;
        const int64_t waves = (items + G - 1) / G;
        const int64_t tiles = (p.n_jt + sp - 1) / sp;
        double cost = (double)waves * (double)(tiles + 2);
        cost += 0.05 * (double)sp * (double)p.n_it * 2.0 * (double)(p.R_pad * (1 + vsplit)) / (double)G / 64.0;
        if (cost < best_cost - 1e-9) { best_cost = cost; best = sp; }
    }
    p.n_split = best;
    const int64_t items = (int64_t)p.n_it * p.n_split;
    p.grid = (int)(items < G ? items : G);
    return p;
}

size_t tp_partial_floats(const TcPlan& p) { return (size_t)p.n_split * p.rv * p.Nr_pad; }

int launch_kmvm_tp(Ctx* ctx, const TcPlan& plan, const OperandLayout& L, const MvmArgs& a, const CUtensorMap& tmA,
                   const CUtensorMap& tmB, const CUtensorMap& tmV, const float* outscale, float* partial,
                   const uint32_t* mask, cudaStream_t s, MvmParts* parts) {
    TpParams prm;
    prm.n_ip = plan.n_it;
    prm.n_jt = plan.n_jt;
    prm.n_split = plan.n_split;
    prm.n_items = plan.n_it * plan.n_split;
    prm.k_pad = plan.k_pad;
    prm.rv = plan.rv;
    prm.lo_off = L.vsplit ? a.R : 0;
    prm.nrhs = a.R;
    prm.spv = L.fp32_pv ? 1 : 0;
    if (!tp_supported(plan.k_pad, plan.R_pad, L.vsplit)) return GP_ERR_UNSUPPORTED;
    const TpSmem m = tp_smem(plan.k_pad, plan.rv);
    if (m.stages < 2) return GP_ERR_UNSUPPORTED;
    prm.stages = m.stages;
    prm.sm = m;
    prm.diag = a.diag_coef != 0.0f ? 1 : 0;
    prm.ld_part = plan.Nr_pad;
    prm.partial = partial;
    prm.out = a.out;
    prm.ld_out = a.ld_out;
    prm.Nr = a.Nr;
    prm.ld_v = a.Nc;
    prm.outscale = outscale;
    prm.Vnoise = a.Vnoise;
    prm.noise = a.noise + a.diag_coef;
    prm.mask = mask;
    prm.mask_words = (plan.n_jt + 31) / 32;
    prm.err = ctx->dev_err;
    prm.limit_ns = kWaitLimitNs;
    const int bf = (L.prec == GP_PREC_BF16) ? 1 : 0;
    cudaError_t e = cudaErrorInvalidValue;
    const bool hs = L.half_exp != 0;
    if (hs && !(a.kernel == GP_KERNEL_RBF && !bf && !L.psplit && plan.k_pad == 16)) return GP_ERR_UNSUPPORTED;
    prof_begin(ctx, s);
#define GPK_TP_CASE(K)                                                                              \
    case K:                                                                                         \
        if (bf)                                                                                     \
            e = L.psplit ? launch_tp_typed<K, 1, 1>(plan, prm, tmA, tmB, tmV, s)                     \
                         : launch_tp_typed<K, 1, 0>(plan, prm, tmA, tmB, tmV, s);                    \
        else                                                                                        \
            e = L.psplit ? launch_tp_typed<K, 0, 1>(plan, prm, tmA, tmB, tmV, s)                     \
                         : launch_tp_typed<K, 0, 0>(plan, prm, tmA, tmB, tmV, s);                    \
        break;
    const bool spv = L.fp32_pv != 0;
    if (spv && (bf || L.psplit || hs || a.R > 4 || !L.vsplit)) return GP_ERR_UNSUPPORTED;
    if (hs) {
        e = launch_tp_typed<GP_KERNEL_RBF, 0, 0, 1>(plan, prm, tmA, tmB, tmV, s);
    } else if (spv) {
        // accumulators for 1, 2 or 4 columns (3 runs as 4 on a zero fourth row of v)
#define GPK_TP_SPV(K)                                                                            \
    case K:                                                                                      \
        e = a.R == 1 ? launch_tp_typed<K, 0, 0, 0, 1>(plan, prm, tmA, tmB, tmV, s)               \
          : a.R == 2 ? launch_tp_typed<K, 0, 0, 0, 2>(plan, prm, tmA, tmB, tmV, s)               \
                     : launch_tp_typed<K, 0, 0, 0, 4>(plan, prm, tmA, tmB, tmV, s);              \
        break;
        switch (a.kernel) {
            GPK_TP_SPV(GP_KERNEL_RBF)
            GPK_TP_SPV(GP_KERNEL_MATERN32)
            GPK_TP_SPV(GP_KERNEL_MATERN12)
            GPK_TP_SPV(GP_KERNEL_MATERN52)
            default: return GP_ERR_INVALID;
        }
#undef GPK_TP_SPV
    } else switch (a.kernel) {
        GPK_TP_CASE(GP_KERNEL_RBF)
        GPK_TP_CASE(GP_KERNEL_MATERN32)
        GPK_TP_CASE(GP_KERNEL_MATERN12)
        GPK_TP_CASE(GP_KERNEL_MATERN52)
        default: return GP_ERR_INVALID;
    }
#undef GPK_TP_CASE
    prof_end(ctx, s);
    ctx->launches++;
    if (e != cudaSuccess) return GP_ERR_CUDA;
    if (!spv && plan.n_split == 1) return GP_OK;
    if (parts) {
        parts->partial = partial;
        parts->outscale = outscale;
        parts->parts = plan.n_split * (L.vsplit ? 2 : 1);
        parts->ld = plan.Nr_pad;
        parts->noise = a.noise + a.diag_coef;
        return GP_OK;
    }
    // splits times hi and lo rows (times the two column halves of the FP32 value product)
    return launch_split_reduce(ctx, partial, plan.n_split * (L.vsplit ? 2 : 1), plan.Nr_pad, a.Nr, a.R, a.R, outscale, 0.0f,
                               a.noise + a.diag_coef, a.Vnoise, a.Nc, a.out, a.ld_out, s);
}

}  // namespace gpk
