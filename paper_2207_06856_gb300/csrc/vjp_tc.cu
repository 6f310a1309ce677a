// The backward of the kernel MVM on the tensor cores (Sec. 4.3, Eq. approx;
// Sec. 2.2, Eq. gradient): the gradient of the bilinear form
//     q = sum_c u_c^T Ktilde w_c
// with respect to (l_1..l_d, a^2, sigma^2) and X, for RBF, Matern-3/2 and
// Matern-5/2 with FP16 operands and FP32 accumulation.
//
// With H_ij = G_ij + G_ji = sum_c (u_ic w_jc + w_ic u_jc) (symmetric), the
// scaled centred inputs x^_i = (x_i - centre) / l and k' = dk/d(r^2):
//     W'_ij = a^2 k'(r_ij^2) H_ij,  rs_i = sum_j W'_ij,  (W'X^)_im = sum_j W'_ij x^_jm,
//     D_im  = sum_j W'_ij (x^_im - x^_jm) = x^_im rs_i - (W'X^)_im,
//     dq/dx_im    = (2 / l_m) D_im,
//     dq/dl_m     = -(2 / l_m) sum_i x^_im D_im,
//     dq/da^2     = 1/2 sum_ij H_ij k(r_ij^2),
//     dq/dsigma^2 = sum_c u_c^T w_c.
// (sum_ij a^2 k' G_ij (x^_im - x^_jm)^2 = 1/2 sum_ij W'_ij (x^_im - x^_jm)^2 =
// sum_i x^_im D_im, because W' is symmetric.)  So one value product
// W' [X^, 1] per row tile gives every derivative: the backward has the
// forward's shape (flash-attention backward: S and H on the tensor core, the
// elementwise W' in registers, then a second contraction).
//
// Per 128 x 128 tile, on tcgen05 with FP32 accumulators in TMEM:
//   S  = XA_i XB_j^T     (the forward's operands: s = -c^2 r^2 / 2)
//   H  = UW_i WU_j^T     UW = [a_c u | w / a_c], WU = [w / a_c | a_c u] in FP16
//                        (a_c a power of two balancing the column pair; one
//                        global power-of-two scale keeps |entries| <= 1)
//   O += W'_i Xt_j^T     Xt = [x^ hi; 1; x^ lo; 0] rows (the ones row gives rs_i);
//                        N = rv = 16 ceil(2 (d + 1) / 16)
// The epilogue forms W' / (a^2 k'_max) = -phi(s) H (phi = k for RBF, e^-u for
// Matern-3/2, (1 + u) e^-u for Matern-5/2) as FP16 and accumulates sum H k per
// thread.  A slot is 64 columns of a tile: S and H take 64 TMEM columns each, W' is
// written over S in place, and three slots form a ring, so that S and H of the next
// slots and the value product of the last one run behind the epilogue's arithmetic
// (with one 128-column S and H for all sixteen warps the tensor pipe was 43 % active).
// The row tile's operands sit in TMEM too (.ts form; copied from shared memory once
// per item), so a 64-column S or H instruction reads 2 KB of shared memory instead
// of 6 KB and takes 34 cycles instead of 51.
//
// Warps: 0-15 epilogue (warpgroup g: slot parity g & 1, half g >> 1 of its columns),
// 16 TMA producer, 17 S issuer and TMEM owner, 18 H issuer, 19 value-product issuer;
// the epilogue tells the issuers by named barriers (see kmvm_tp.cu).  TMEM: slot b S at
// 128 b, H at 128 b + 64; O at 384; XA_i at 448, UW_i at 480.  Every wait is bounded.
//
// N = 65,536, d = 18 (k_pad 64), 17 columns, RBF: 1.58 ms per launch with one
// 128-column S and H for all warps, 1.18 ms now, against 0.63 of tensor work (760 cycles a
// tile; ex2 takes 512).  What is left is latency: beside four busy warps an issuer's
// instruction waits its turn, and a slot passes S / H, epilogue and value product in sequence.
#include "gpk_internal.cuh"
#include "ptx.cuh"
#include "kfun.cuh"

#include <math.h>

namespace gpk {

namespace {

constexpr int kBM = 128;
constexpr int kBN = 128;
constexpr int kEpiWarps = 16;
constexpr int kThreads = (kEpiWarps + 4) * 32;
constexpr int kTmaWarp = kEpiWarps;
constexpr int kShWarp = kEpiWarps + 1;    // S issuer (TMEM owner), then the H issuer
constexpr int kOWarp = kEpiWarps + 3;
constexpr int kMaxStages = 4;
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kRing = 3;             // slots of 64 columns
constexpr uint32_t kColO = 384, kColXA = 448, kColUW = 480;
constexpr uint32_t kBarThreads = 9 * 32;  // 8 epilogue warps and one issuer (kBarA: two)
constexpr uint32_t kBarA = 1, kBarW = 2;  // row operands in TMEM; W' of slot b stored (kBarW + b)
constexpr int kMaxSmemBytes = 227 * 1024;

struct VjpSmem {
    uint32_t xbytes, hbytes, vbytes, stage_bytes, xi_bytes;
    int stages;
    uint32_t total;
};

__host__ __device__ inline VjpSmem vjp_smem(int k_pad, int kh, int rv) {
    VjpSmem m;
    m.xbytes = (uint32_t)kBM * (uint32_t)k_pad * 2u;
    m.hbytes = (uint32_t)kBM * (uint32_t)kh * 2u;
    m.vbytes = 2u * (uint32_t)rv * 128u;                 // two 64-column K-blocks of rv rows
    m.stage_bytes = m.xbytes + m.hbytes + m.vbytes;
    m.xi_bytes = m.xbytes + m.hbytes;
    const uint32_t fixed = 1024u + 2u * m.xi_bytes;
    m.stages = 0;
    for (int s = kMaxStages; s >= 2; --s)
        if (fixed + (uint32_t)s * m.stage_bytes <= (uint32_t)kMaxSmemBytes - 512u) { m.stages = s; break; }
    m.total = fixed + (uint32_t)m.stages * m.stage_bytes;
    return m;
}

struct VjpParams {
    int n_it, n_jt, n_split, n_items;
    int k_pad, kh, rv;       // S contraction width, H contraction width (2 R_pad), O width
    int stages;
    VjpSmem sm;
    int64_t N_pad;
    float* part;             // [n_split][rv][N_pad]: raw O columns
    double* hk;              // [gridDim.x]: per-CTA sum of H k
    int* err;
    uint64_t limit_ns;
};

struct VjpBarriers {
    uint64_t full[kMaxStages];
    uint64_t empty[kMaxStages];
    uint64_t xi_full[2];
    uint64_t xi_empty[2];
    uint64_t sh_full[kRing];
    uint64_t w_empty[kRing];    // W' consumed: S and H of a later slot may overwrite the buffer
    uint64_t o_full;
    uint64_t o_empty;
    uint64_t drain[3];
};

__device__ __forceinline__ void record_error(int* err, int code) { atomicCAS(err, 0, code); }

__device__ __forceinline__ void item_range(const VjpParams& p, int item, int& it, int& sp, int& j0, int& j1) {
    // 32-bit: n_split <= 16 and n_jt <= 2^24
    const uint32_t q = (uint32_t)item / (uint32_t)p.n_it;
    sp = (int)q;
    it = item - sp * p.n_it;
    j0 = (int)(q * (uint32_t)p.n_jt / (uint32_t)p.n_split);
    j1 = (int)((q + 1u) * (uint32_t)p.n_jt / (uint32_t)p.n_split);
}

__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, uint64_t limit_ns) {
    return __all_sync(0xffffffffu, ptx::mbar_wait(bar, parity, limit_ns));
}

__device__ __forceinline__ uint32_t swz_code(uint32_t row_bytes) {
    return row_bytes == 32u ? 6u : (row_bytes == 64u ? 4u : 2u);
}

// ---- TMA producer (one thread) ------------------------------------------------
__device__ void vjp_producer(const VjpParams& p, const CUtensorMap* tmA, const CUtensorMap* tmB,
                             const CUtensorMap* tmUW, const CUtensorMap* tmWU, const CUtensorMap* tmXt,
                             VjpBarriers& bars, uint8_t* sSt, uint8_t* sXi, const VjpSmem& m) {
    uint32_t fills = 0, xi_loads = 0;
    bool ok = true;
    int ic = 0;
    const uint32_t S = (uint32_t)p.stages;
    const uint32_t vbox = (uint32_t)p.rv * 128u;
#pragma unroll 1
    for (int item = blockIdx.x; item < p.n_items; item += gridDim.x, ++ic) {
        int it, sp, j0, j1;
        item_range(p, item, it, sp, j0, j1);
        const int xb = ic & 1;
        if (ic >= 2 && !ptx::mbar_wait(&bars.xi_empty[xb], ((ic >> 1) - 1) & 1, p.limit_ns)) { ok = false; break; }
        uint8_t* sX = sXi + (uint32_t)xb * m.xi_bytes;
        ptx::mbar_arrive_expect_tx(&bars.xi_full[xb], m.xi_bytes);
        ptx::tma_load_2d(sX, tmA, &bars.xi_full[xb], 0, it * kBM);
        ptx::tma_load_2d(sX + m.xbytes, tmUW, &bars.xi_full[xb], 0, it * kBM);
        ++xi_loads;
#pragma unroll 1
        for (int jt = j0; jt < j1; ++jt) {
            const uint32_t st = fills % S, u = fills / S;
            if (u > 0 && !ptx::mbar_wait_sleep(&bars.empty[st], (u - 1) & 1, p.limit_ns)) { ok = false; break; }
            uint8_t* sx = sSt + st * m.stage_bytes;
            ptx::mbar_arrive_expect_tx(&bars.full[st], m.stage_bytes);
            ptx::tma_load_2d(sx, tmB, &bars.full[st], 0, jt * kBN);
            ptx::tma_load_2d(sx + m.xbytes, tmWU, &bars.full[st], 0, jt * kBN);
            ptx::tma_load_2d(sx + m.xbytes + m.hbytes, tmXt, &bars.full[st], jt * kBN, 0);
            ptx::tma_load_2d(sx + m.xbytes + m.hbytes + vbox, tmXt, &bars.full[st], jt * kBN + 64, 0);
            ++fills;
        }
        if (!ok) break;
    }
    if (!ok) {
        record_error(p.err, DEV_TIMEOUT);
        // every copy this thread issued lands before the CTA can exit
        const uint32_t first = fills > S ? fills - S : 0;
        for (uint32_t f = first; f < fills; ++f) ptx::mbar_wait(&bars.full[f % S], (f / S) & 1, p.limit_ns);
        for (uint32_t q = xi_loads > 2 ? xi_loads - 2 : 0; q < xi_loads; ++q)
            ptx::mbar_wait(&bars.xi_full[q & 1], (q >> 1) & 1, p.limit_ns);
    }
}

// ---- S and H issuers (two converged warps) ----------------------------------------
// K-steps of 16 of a 64-column product and its commit: A from TMEM, B rows of
// `row` bytes (32, 64 or 128) at descriptor word lB.
__device__ __forceinline__ void vjp_product(uint32_t tD, uint32_t tA, uint32_t lB, uint32_t row, uint32_t hi, uint32_t id,
                                            uint32_t bar) {
    if (row == 128u) {
        ptx::mma_f16_ts4_elect<8, 16, 24>(tD, tA, lB, hi, id, 0u, bar);
    } else {
#pragma unroll 1
        for (uint32_t k = 0; k < row; k += 32u)
            ptx::mma_f16_ts_elect(tD, tA + k / 4u, ((uint64_t)hi << 32) | (lB + k / 16u), id, k > 0 ? 1u : 0u);
        ptx::mma_commit_elect(bar);
    }
}

// S (which = 0) or H (which = 1) of each slot once the value product of the slot
// kRing before it has completed and the stage has landed (one probe: even lanes look
// at one barrier, odd lanes at the other); an item's first slot also waits for the row
// operands in TMEM.  One warp issuing both spent 600-800 cycles a slot on probes,
// descriptors and instructions, against 380 of tensor work.  A bounded wait that runs
// out makes the role go on without waits or tensor work, meeting its named barriers.
__device__ void vjp_mma_sh(const VjpParams& p, VjpBarriers& bars, const uint8_t* sSt, const VjpSmem& m, uint32_t tmem,
                           uint32_t which) {
    const uint32_t row = (uint32_t)(which ? p.kh : p.k_pad) * 2u;
    const uint32_t hi = ptx::smem_desc_hi(8u * row, swz_code(row));
    const uint32_t id = ptx::idesc_f16(kBM, 64, 0);
    const uint32_t lB0 = ptx::smem_desc_lo(ptx::smem_u32(sSt) + (which ? m.xbytes : 0u));
    const uint32_t sh_full = ptx::smem_u32(&bars.sh_full[0]);
    const uint32_t tA = tmem + (which ? kColUW : kColXA), tD = tmem + 64u * which;
    const bool odd = threadIdx.x & 1;
    uint32_t st = 0, ph = 0, b = 0, bph = 1;   // bph: parity of the buffer's last release (first round: passes at once)
    bool ok = true;
#pragma unroll 1
    for (int item = blockIdx.x; item < p.n_items; item += gridDim.x) {
        int it, sp, j0, j1;
        item_range(p, item, it, sp, j0, j1);
        ptx::bar_sync(kBarA, kBarThreads + 32u);
#pragma unroll 1
        for (int jt = j0; jt < j1; ++jt) {
            const uint32_t lB = lB0 + st * (m.stage_bytes >> 4);
#pragma unroll 1
            for (uint32_t h = 0; h < 2; ++h) {
                ok = ok && __all_sync(0xffffffffu, ptx::mbar_wait(odd ? &bars.full[st] : &bars.w_empty[b],
                                                                  odd ? ph : bph, p.limit_ns));
                if (ok) {
                    ptx::tc_fence_after();
                    vjp_product(tD + b * 128u, tA, lB + h * 4u * row, row, hi, id, sh_full + 8u * b);
                }
                if (++b == kRing) { b = 0; bph ^= 1u; }
            }
            if (++st == (uint32_t)p.stages) { st = 0; ph ^= 1u; }
        }
    }
    ptx::mma_commit_elect(&bars.drain[which]);
    warp_wait(&bars.drain[which], 0, p.limit_ns);
    if (!ok && (threadIdx.x & 31) == 0) record_error(p.err, DEV_TIMEOUT);
}

// ---- value-product issuer (one converged warp) ------------------------------------
// O += W' Xt_j^T for each slot once its W' is stored; then the slot's buffer and,
// after the tile's second slot, the stage are released.  O is handed to the
// epilogue at the end of an item.
__device__ void vjp_mma_o(const VjpParams& p, VjpBarriers& bars, const uint8_t* sSt, const VjpSmem& m,
                          uint32_t tmem) {
    const uint32_t hi_v = ptx::smem_desc_hi(1024u, 2u);
    const uint32_t id = ptx::idesc_f16(kBM, p.rv, 0);
    const uint32_t lV0 = ptx::smem_desc_lo(ptx::smem_u32(sSt) + m.xbytes + m.hbytes);
    const uint32_t kb = (uint32_t)p.rv * 8u;   // a 64-column K-block in 16-byte units
    const uint32_t w_empty = ptx::smem_u32(&bars.w_empty[0]);
    uint32_t st = 0, ph = 0, b = 0;
    int ic = 0;
    bool ok = true;
#pragma unroll 1
    for (int item = blockIdx.x; item < p.n_items; item += gridDim.x, ++ic) {
        int it, sp, j0, j1;
        item_range(p, item, it, sp, j0, j1);
        if (ic > 0) ok = ok && warp_wait(&bars.o_empty, (ic - 1) & 1, p.limit_ns);
#pragma unroll 1
        for (int jt = j0; jt < j1; ++jt) {
            ok = ok && warp_wait(&bars.full[st], ph, p.limit_ns);   // Xt_j: landed for S
            const uint32_t lV = lV0 + st * (m.stage_bytes >> 4);
#pragma unroll 1
            for (uint32_t h = 0; h < 2; ++h) {
                ptx::bar_sync(kBarW + b, kBarThreads);
                if (ok) {
                    ptx::tc_fence_after();
                    ptx::mma_f16_ts4_elect<8, 32, 40>(tmem + kColO, tmem + b * 128u, lV + h * kb, hi_v, id,
                                                      (jt > j0 || h > 0) ? 1u : 0u, w_empty + 8u * b);
                }
                if (++b == kRing) b = 0;
            }
            if (ok) ptx::mma_commit_elect(&bars.empty[st]);     // the stage's operands are consumed
            if (++st == (uint32_t)p.stages) { st = 0; ph ^= 1u; }
        }
        if (ok) ptx::mma_commit_elect(&bars.o_full);
    }
    ptx::mma_commit_elect(&bars.drain[2]);
    warp_wait(&bars.drain[2], 0, p.limit_ns);
    if (!ok && (threadIdx.x & 31) == 0) record_error(p.err, DEV_TIMEOUT);
}

// ---- epilogue: W' = -phi(s) H in FP16, sum H k --------------------------------------
template <int KIND>
__device__ __forceinline__ void wprime(float s, float h, float& w, float& hk) {
    if constexpr (KIND == GP_KERNEL_RBF) {
        const float k = ptx::ex2(s);                      // s = -log2(e) r^2 / 2
        w = -k * h;                                       // k' = -k / 2, k'_max = 1/2
        hk = h * k;
    } else {
        const float u = ptx::sqrt_approx(fmaxf(-s, 0.0f));   // u = sqrt3 r (Matern-3/2), sqrt5 r (5/2)
        const float e = ptx::ex2(-kLog2e * u);
        if constexpr (KIND == GP_KERNEL_MATERN32) {
            w = -e * h;                                   // k' = -(3/2) e^-u, k'_max = 3/2
            hk = h * fmaf(u, e, e);
        } else {
            const float pu = 1.0f + u;
            w = -pu * e * h;                              // k' = -(5/6)(1 + u) e^-u, k'_max = 5/6
            hk = h * (fmaf(u * u, 1.0f / 3.0f, pu) * e);
        }
    }
}

// A row operand of an item from its swizzled shared-memory tile (rows of `row`
// bytes) into TMEM: this thread's row, 16-byte chunks in K order, 4 columns each.
__device__ __forceinline__ void vjp_row_to_tmem(uint32_t sT, uint32_t row, uint32_t r, uint32_t tA) {
    const uint32_t mask = row / 16u - 1u;   // chunks per row - 1 = the swizzle's address bits
    for (uint32_t c = 0; c < row / 16u; c += 2) {
        uint32_t v[8];
#pragma unroll
        for (uint32_t u = 0; u < 2; ++u) {
            const uint32_t off = r * row + (c + u) * 16u;
            const uint32_t phys = off ^ (((off >> 7) & mask) << 4);
            asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(v[4 * u]), "=r"(v[4 * u + 1]), "=r"(v[4 * u + 2]), "=r"(v[4 * u + 3])
                         : "r"(sT + phys));
        }
        ptx::tmem_st8(tA + c * 4u, v);
    }
}

template <int KIND>
__device__ void vjp_epilogue(const VjpParams& p, VjpBarriers& bars, const uint8_t* sXi, const VjpSmem& m, uint32_t tmem,
                             int wg, int wq, int lane, double* red) {
    const int pr = wg & 1, ch = wg >> 1;              // slot parity (half of a tile), half of its 64 columns
    const uint32_t lane_off = (uint32_t)(wq * 32) << 16;
    uint32_t b = (uint32_t)pr, ph = 0;                // ring slot of this warp's next slot and its fill parity
    int ic = 0;
    bool ok = true;
    double acc = 0.0;
#pragma unroll 1
    for (int item = blockIdx.x; item < p.n_items; item += gridDim.x, ++ic) {
        int it, sp, j0, j1;
        item_range(p, item, it, sp, j0, j1);
        if (pr == 0) {
            // warpgroup 0: XA_i, warpgroup 2: UW_i.  The products of the last item that read them are done
            // (its O was complete).
            ok = ok && warp_wait(&bars.xi_full[ic & 1], (ic >> 1) & 1, p.limit_ns);
            const uint32_t sX = ptx::smem_u32(sXi) + (uint32_t)(ic & 1) * m.xi_bytes;
            const uint32_t r = (uint32_t)(wq * 32 + lane);
            if (ch == 0) vjp_row_to_tmem(sX, (uint32_t)p.k_pad * 2u, r, tmem + lane_off + kColXA);
            else vjp_row_to_tmem(sX + m.xbytes, (uint32_t)p.kh * 2u, r, tmem + lane_off + kColUW);
            ptx::tmem_wait_st();
            ptx::tc_fence_before();
            ptx::bar_arrive(kBarA, kBarThreads + 32u, ok);
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&bars.xi_empty[ic & 1]);
        }
#pragma unroll 1
        for (int jt = j0; jt < j1; ++jt) {
            ok = ok && warp_wait(&bars.sh_full[b], ph, p.limit_ns);
            ptx::tc_fence_after();
            const uint32_t tS = tmem + lane_off + b * 128u + (uint32_t)ch * 32u;
            uint32_t rs[32], rh[32];
            ptx::tmem_ld32(tS, rs);
            ptx::tmem_ld32(tS + 64u, rh);
            ptx::tmem_wait_ld();
            ptx::tmem_reg_fence(rs);
            ptx::tmem_reg_fence(rh);
            uint32_t pk[16];
            float a = 0.0f;
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                float w0, w1, h0, h1;
                wprime<KIND>(__uint_as_float(rs[2 * e]), __uint_as_float(rh[2 * e]), w0, h0);
                wprime<KIND>(__uint_as_float(rs[2 * e + 1]), __uint_as_float(rh[2 * e + 1]), w1, h1);
                a += h0 + h1;
                __half2 hv = __floats2half2_rn(w0, w1);
                pk[e] = *reinterpret_cast<uint32_t*>(&hv);
            }
            ptx::tmem_st16(tS, pk);
            ptx::tmem_wait_st();
            ptx::tc_fence_before();
            ptx::bar_arrive(kBarW + b, kBarThreads, ok);
            acc += (double)a;   // FP64 is slow here: behind the arrival
            b += 2;
            if (b >= kRing) { b -= kRing; ph ^= 1u; }
        }
        // O read-out in chunks of 8 columns, dealt to the warpgroups
        ok = ok && warp_wait(&bars.o_full, ic & 1, p.limit_ns);
        ptx::tc_fence_after();
        const int64_t row = (int64_t)it * kBM + wq * 32 + lane;
#pragma unroll 1
        for (int c0 = 8 * wg; c0 < p.rv; c0 += 32) {
            float* dst = p.part + ((int64_t)sp * p.rv + c0) * p.N_pad + row;
            uint32_t o[8];
            ptx::tmem_ld8(tmem + lane_off + kColO + (uint32_t)c0, o);
            ptx::tmem_wait_ld();
            ptx::tmem_reg_fence(o);
#pragma unroll
            for (int c = 0; c < 8; ++c) dst[(int64_t)c * p.N_pad] = __uint_as_float(o[c]);
        }
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(&bars.o_empty);
    }
    if (!ok && lane == 0) record_error(p.err, DEV_TIMEOUT);
    // per-CTA sum of H k in a fixed order: warp shuffle tree, then the warps in order
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) red[wg * 4 + wq] = acc;
}

template <int KIND>
__global__ void __launch_bounds__(kThreads, 1)
kvjp_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
               const __grid_constant__ CUtensorMap tmUW, const __grid_constant__ CUtensorMap tmWU,
               const __grid_constant__ CUtensorMap tmXt, const VjpParams p) {
    extern __shared__ uint8_t dsm[];
    __shared__ VjpBarriers bars;
    __shared__ uint32_t tmem_slot;
    __shared__ double red[kEpiWarps];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(dsm) + 1023) & ~uintptr_t(1023));
    const VjpSmem& m = p.sm;
    uint8_t* sSt = base;
    uint8_t* sXi = base + (uint32_t)p.stages * m.stage_bytes;
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // warp-uniform
    if (threadIdx.x == 0) {
#pragma unroll 1
        for (int s = 0; s < kMaxStages; ++s) {
            ptx::mbar_init(&bars.full[s], 1);
            ptx::mbar_init(&bars.empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            ptx::mbar_init(&bars.xi_full[b], 1);
            ptx::mbar_init(&bars.xi_empty[b], 8);         // the warps that copy the row operands
        }
        for (uint32_t b = 0; b < 3; ++b) ptx::mbar_init(&bars.drain[b], 1);
        for (uint32_t b = 0; b < kRing; ++b) {
            ptx::mbar_init(&bars.sh_full[b], 2);          // the S and the H issuer
            ptx::mbar_init(&bars.w_empty[b], 1);
        }
        ptx::mbar_init(&bars.o_full, 1);
        ptx::mbar_init(&bars.o_empty, kEpiWarps);
        ptx::fence_mbar_init();
    }
    if (warp == kTmaWarp && lane == 0) {
        ptx::tma_prefetch_desc(&tmA);
        ptx::tma_prefetch_desc(&tmB);
        ptx::tma_prefetch_desc(&tmUW);
        ptx::tma_prefetch_desc(&tmWU);
        ptx::tma_prefetch_desc(&tmXt);
    }
    if (warp == kShWarp) ptx::tmem_alloc(&tmem_slot, kTmemCols);
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = tmem_slot;
    if (warp == kTmaWarp) {
        if (lane == 0) vjp_producer(p, &tmA, &tmB, &tmUW, &tmWU, &tmXt, bars, sSt, sXi, m);
        __syncwarp();
    } else if (warp == kShWarp || warp == kShWarp + 1) {
        vjp_mma_sh(p, bars, sSt, m, tmem, (uint32_t)(warp - kShWarp));
    } else if (warp == kOWarp) {
        vjp_mma_o(p, bars, sSt, m, tmem);
    } else {
        vjp_epilogue<KIND>(p, bars, sXi, m, tmem, warp >> 2, warp & 3, lane, red);
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kEpiWarps; ++w) t += red[w];
        p.hk[blockIdx.x] = t;
    }
    if (warp == kShWarp) ptx::tmem_dealloc(tmem, kTmemCols);
}

// ---- operand preparation and the final reductions ----------------------------------
// scales[c] = a_c (power of two balancing max|u_c| and max|w_c|), scales[rp] = g:
// the power of two that brings every entry of [a u | w / a] to |.| <= 1.
__global__ void uw_scales_kernel(const unsigned* __restrict__ cmu, const unsigned* __restrict__ cmw, int R, int rp,
                                 float* __restrict__ scales, int* err) {
    __shared__ float mx[32];
    const int c = threadIdx.x;   // one warp, R <= 32
    float a = 1.0f, m = 0.0f;
    if (c < R) {
        const float mu = __uint_as_float(cmu[c]), mw = __uint_as_float(cmw[c]);
        if (!(mu <= 3.0e38f) || !(mw <= 3.0e38f)) {
            atomicCAS(err, 0, (int)DEV_NONFINITE);
        } else {
            if (mu > 0.0f && mw > 0.0f) a = exp2f(rintf(0.5f * log2f(mw / mu)));
            m = fmaxf(a * mu, mw / a);
        }
        scales[c] = a;
    }
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (c == 0) {
        float g = 1.0f;
        if (m > 0.0f) {
            int e;
            frexpf(m, &e);            // m = f 2^e, f in [1/2, 1)
            g = ldexpf(1.0f, -e);     // m g < 1
        }
        scales[rp] = g;
    }
    (void)mx;
}

// UW[i] = g [a_c u_ic | w_ic / a_c], WU[i] = g [w_ic / a_c | a_c u_ic] in FP16 (rows i < N_pad,
// zero beyond N and beyond R in each half); U, W: R x N (column c at c * N).
__global__ void uw_prep_kernel(const float* __restrict__ U, const float* __restrict__ W, int64_t N, int64_t N_pad,
                               int R, int rp, const float* __restrict__ scales, __half* __restrict__ UW,
                               __half* __restrict__ WU) {
    const int kh = 2 * rp;
    const float g = scales[rp];
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < N_pad * kh;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = e / kh;
        const int col = (int)(e % kh);
        const int c = col < rp ? col : col - rp;
        float uw = 0.0f, wu = 0.0f;
        if (i < N && c < R) {
            const float a = scales[c];
            const float u = U[(int64_t)c * N + i] * a * g, w = W[(int64_t)c * N + i] / a * g;
            uw = col < rp ? u : w;
            wu = col < rp ? w : u;
        }
        UW[e] = __float2half_rn(uw);
        WU[e] = __float2half_rn(wu);
    }
}

__device__ __forceinline__ float decode_order(unsigned s) {
    return __uint_as_float((s & 0x80000000u) ? (s & 0x7FFFFFFFu) : ~s);
}

// Vb (d + 1 columns of N, FP32): x^_m = (x_m - centre_m) / l_m, then a column of ones.
__global__ void vb_prep_kernel(const float* __restrict__ X, int64_t N, int d, ScaleVec il,
                               const unsigned* __restrict__ bb, float* __restrict__ Vb) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < N * (d + 1);
         e += (int64_t)gridDim.x * blockDim.x) {
        const int m = (int)(e / N);
        const int64_t i = e % N;
        if (m < d) {
            const float centre = 0.5f * (decode_order(~bb[m]) + decode_order(bb[d + m]));
            Vb[e] = (X[i * d + m] - centre) * il.v[m];
        } else {
            Vb[e] = 1.0f;
        }
    }
}

// Per row i < N: O_c = sum_s (part[s][c][i] + part[s][rx + c][i]) xs_c (hi + lo rows of Xt),
// rs_i = O_d, D_im = x^_im rs_i - O_m; gX_im = (2 / l_m) F D_im; per block sum_i x^_im D_im (FP64).
// F = a^2 k'_max / g^2 undoes the storage scale of W'.
__global__ void __launch_bounds__(256)
vjp_finish_kernel(const float* __restrict__ part, int n_split, int rv, int64_t N_pad, const float* __restrict__ xs,
                  const float* __restrict__ Vb, int64_t N, int d, ScaleVec two_over_l, float a2kp,
                  const float* __restrict__ scales, int rp, float* __restrict__ gX, double* __restrict__ lpart) {
    const int rx = d + 1;
    const float g = scales[rp];
    const float F = a2kp / (g * g);
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double lsum[32];
#pragma unroll
    for (int m = 0; m < 32; ++m) lsum[m] = 0.0;
    if (i < N) {
        float rs = 0.0f;
        for (int s = 0; s < n_split; ++s)
            rs += part[((int64_t)s * rv + d) * N_pad + i] + part[((int64_t)s * rv + rx + d) * N_pad + i];
        rs *= xs[d];
#pragma unroll
        for (int m = 0; m < 32; ++m) {
            if (m < d) {
                float o = 0.0f;
                for (int s = 0; s < n_split; ++s)
                    o += part[((int64_t)s * rv + m) * N_pad + i] + part[((int64_t)s * rv + rx + m) * N_pad + i];
                const float xh = Vb[(int64_t)m * N + i];
                const float D = fmaf(xh, rs, -o * xs[m]);
                if (gX) gX[i * d + m] = two_over_l.v[m] * F * D;
                lsum[m] = (double)xh * (double)D;
            }
        }
    }
    // Warp sums of the 32 values by a transposing butterfly: at distance o each lane
    // hands over the half of its values whose index differs from its own in bit o,
    // so 31 FP64 additions replace 32 x 5 (the same tree per value) and lane m ends
    // with the sum of value m.
    __shared__ double red[8][32];
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const bool up = (l & o) != 0;
#pragma unroll
        for (int m = 0; m < o; ++m) {
            const double keep = up ? lsum[m + o] : lsum[m], give = up ? lsum[m] : lsum[m + o];
            lsum[m] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    red[w][l] = lsum[0];
    __syncthreads();
    if (threadIdx.x < 32) {
        double t = 0.0;
        for (int q = 0; q < 8; ++q) t += red[q][threadIdx.x];
        lpart[(int64_t)blockIdx.x * 32 + threadIdx.x] = t * (double)F;
    }
}

// out[s] = sum_b part[b * stride + s], one warp per slot s (lanes stride over b,
// then a shuffle tree: a fixed order).
__global__ void __launch_bounds__(32)
sum_rows_kernel(const double* __restrict__ part, int nb, int stride, double* __restrict__ out) {
    const int s = blockIdx.x, l = threadIdx.x;
    double t = 0.0;
#pragma unroll 4
    for (int b = l; b < nb; b += 32) t += part[(int64_t)b * stride + s];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (l == 0) out[s] = t;
}

// part[c * gridDim.x + blk] = the block's part of u_c^T w_c in FP64 (fixed-order tree)
__global__ void __launch_bounds__(256)
coldot2_kernel(const float* __restrict__ U, const float* __restrict__ W, int64_t N, double* __restrict__ part) {
    const int c = blockIdx.y;
    double acc = 0.0;
#pragma unroll 4
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < N; i += (int64_t)gridDim.x * 256)
        acc = fma((double)U[(int64_t)c * N + i], (double)W[(int64_t)c * N + i], acc);
    __shared__ double r[8];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) r[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int q = 0; q < 8; ++q) t += r[q];
        part[(int64_t)c * gridDim.x + blockIdx.x] = t;
    }
}

float kprime_max(int kernel) {
    return kernel == GP_KERNEL_RBF ? 0.5f : (kernel == GP_KERNEL_MATERN32 ? 1.5f : 5.0f / 6.0f);
}

CUtensorMapSwizzle swz_for(uint32_t row_bytes) {
    return row_bytes == 32 ? CU_TENSOR_MAP_SWIZZLE_32B
                           : (row_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B);
}

}  // namespace

bool vjp_tc_supported(const gp_hyp_t* hyp, int R) {
    if (hyp->kernel == GP_KERNEL_MATERN12) return false;   // k' ~ 1/r: singular at coincident points
    if (hyp->d > 31 || R > 32) return false;
    const OperandLayout L = make_layout(hyp->d, GP_PREC_FP16, hyp->d > 12 ? 1 : 0, 1, 0);
    return L.k_pad != 0 && L.k_pad <= 64;
}

namespace {

constexpr int kDotBlocks = 16;   // blocks per column of the sigma^2 dots

struct VjpPlan {
    int n_it, n_jt, n_split, grid, rp, kh, rx, rv;
    int64_t N_pad, Nc_pad;
    int nblk_f;
};

VjpPlan vjp_plan(const Ctx* ctx, const KOp& op, int64_t N, int d, int R) {
    VjpPlan p;
    p.N_pad = op.tp.Nr_pad;
    p.Nc_pad = op.tp.Nc_pad;
    p.n_it = (int)((N + kBM - 1) / kBM);
    p.n_jt = (int)(p.Nc_pad / kBN);
    p.rp = R <= 16 ? 16 : 32;
    p.kh = 2 * p.rp;
    p.rx = d + 1;                                  // rows of Xt per part: hi, then lo
    p.rv = ((2 * p.rx + 15) / 16) * 16;
    const int G = ctx->num_sms > 0 ? ctx->num_sms : 1;
    // column split minimising the busiest CTA's tiles (+ about two tiles of per-item cost)
    int best = 1;
    double best_cost = 1e300;
    const int max_split = p.n_jt < 16 ? p.n_jt : 16;
    for (int sp = 1; sp <= max_split; ++sp) {
        const int64_t items = (int64_t)p.n_it * sp;
        const int64_t waves = (items + G - 1) / G;
        const int64_t tiles = (p.n_jt + sp - 1) / sp;
        const double cost = (double)waves * (double)(tiles + 2);
        if (cost < best_cost - 1e-9) { best_cost = cost; best = sp; }
    }
    p.n_split = best;
    const int64_t items = (int64_t)p.n_it * p.n_split;
    p.grid = (int)(items < G ? items : G);
    p.nblk_f = (int)((N + 255) / 256);
    return p;
}

template <class C>
void vjp_tc_layout(C& c, const VjpPlan& p, int64_t N, int d, int R) {
    c.template take<__half>((size_t)p.N_pad * p.kh);     // UW
    c.template take<__half>((size_t)p.N_pad * p.kh);     // WU
    c.template take<unsigned>(64);                        // column maxima of U, W, Vb
    c.template take<unsigned>(64);
    c.template take<unsigned>(64);
    c.template take<float>(64);                           // a_c, g
    c.template take<float>((size_t)N * (d + 1));          // Vb
    c.template take<__half>((size_t)p.rv * p.Nc_pad);     // Xt
    c.template take<float>(64);                           // column scales of Xt
    c.template take<float>((size_t)p.n_split * p.rv * p.N_pad);   // O partials
    c.template take<double>((size_t)p.grid);              // per-CTA sum H k
    c.template take<double>((size_t)p.nblk_f * 32);       // per-block lengthscale sums
    c.template take<double>(64);                          // sums
    c.template take<double>((size_t)R * kDotBlocks);      // column dots, per block
}

}  // namespace

size_t vjp_tc_workspace(const Ctx* ctx, const gp_hyp_t* hyp, int64_t N, int R) {
    KOp op;
    const size_t kw = kop_workspace(ctx, hyp, N, N, 1, GP_PREC_FP16, true);
    if (kw == 0) return 0;
    // the plan only needs the padded sizes, which depend on N alone
    op.tp = tp_plan(ctx, N, N, 1, 16, 1);
    const VjpPlan p = vjp_plan(ctx, op, N, hyp->d, R);
    WsCounter c;
    vjp_tc_layout(c, p, N, hyp->d, R);
    return kw + c.off;
}

int vjp_tc_run(Ctx* ctx, WsCarver& wc, const gp_hyp_t* hyp, const float* X, int64_t N, const float* U,
               const float* W, int R, double* grad_theta_host, float* gX_dev, cudaStream_t s) {
    const int d = hyp->d;
    KOp op;
    GPK_TRY(kop_prepare(ctx, wc, op, hyp, X, N, X, N, 1, GP_PREC_FP16, s));
    if (op.tp.engine != 1 || op.lay.k_pad > 64) return GP_ERR_UNSUPPORTED;
    const VjpPlan pl = vjp_plan(ctx, op, N, d, R);
    __half* UW = wc.take<__half>((size_t)pl.N_pad * pl.kh);
    __half* WU = wc.take<__half>((size_t)pl.N_pad * pl.kh);
    unsigned* cmu = wc.take<unsigned>(64);
    unsigned* cmw = wc.take<unsigned>(64);
    unsigned* cmv = wc.take<unsigned>(64);
    float* scales = wc.take<float>(64);
    float* Vb = wc.take<float>((size_t)N * (d + 1));
    __half* Xt = wc.take<__half>((size_t)pl.rv * pl.Nc_pad);
    float* xs = wc.take<float>(64);
    float* part = wc.take<float>((size_t)pl.n_split * pl.rv * pl.N_pad);
    double* hk = wc.take<double>((size_t)pl.grid);
    double* lpart = wc.take<double>((size_t)pl.nblk_f * 32);
    double* sums = wc.take<double>(64);
    double* dots = wc.take<double>((size_t)R * kDotBlocks);
    if (!wc.ok) return GP_ERR_WORKSPACE;

    // H operands: balanced, globally scaled FP16 copies of [u | w] and [w | u]
    GPK_TRY(launch_v_colmax(ctx, U, N, R, cmu, s));
    GPK_TRY(launch_v_colmax(ctx, W, N, R, cmw, s));
    uw_scales_kernel<<<1, 32, 0, s>>>(cmu, cmw, R, pl.rp, scales, ctx->dev_err);
    int64_t g1 = (pl.N_pad * pl.kh + 255) / 256;
    if (g1 > 8192) g1 = 8192;
    uw_prep_kernel<<<(unsigned)g1, 256, 0, s>>>(U, W, N, pl.N_pad, R, pl.rp, scales, UW, WU);
    // value-product operand: [x^ (centred, / l), 1] as hi + lo FP16 rows
    ScaleVec il;
    for (int k = 0; k < 64; ++k) il.v[k] = k < d ? (float)(1.0 / (double)hyp->lengthscale[k]) : 0.0f;
    int64_t g2 = (N * (d + 1) + 255) / 256;
    if (g2 > 8192) g2 = 8192;
    vb_prep_kernel<<<(unsigned)g2, 256, 0, s>>>(X, N, d, il, op.bbox, Vb);
    ctx->launches += 3;
    if (cudaGetLastError() != cudaSuccess) return GP_ERR_CUDA;
    GPK_TRY(launch_v_colmax(ctx, Vb, N, d + 1, cmv, s));
    GPK_TRY(launch_v_cast(ctx, GP_PREC_FP16, 0, 1, Vb, N, pl.Nc_pad, d + 1, pl.rx, pl.rv, cmv, 1.0, Xt, xs, s));

    CUtensorMap tmUW, tmWU, tmXt;
    const uint32_t hrow = (uint32_t)pl.kh * 2u;
    GPK_TRY(encode_tmap_2d(&tmUW, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, UW, pl.kh, pl.N_pad, hrow, pl.kh, 128,
                           swz_for(hrow)));
    GPK_TRY(encode_tmap_2d(&tmWU, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, WU, pl.kh, pl.N_pad, hrow, pl.kh, 128,
                           swz_for(hrow)));
    GPK_TRY(encode_tmap_2d(&tmXt, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, Xt, pl.Nc_pad, pl.rv, pl.Nc_pad * 2, 64,
                           (uint32_t)pl.rv, CU_TENSOR_MAP_SWIZZLE_128B));

    VjpParams prm;
    prm.n_it = pl.n_it;
    prm.n_jt = pl.n_jt;
    prm.n_split = pl.n_split;
    prm.n_items = pl.n_it * pl.n_split;
    prm.k_pad = op.lay.k_pad;
    prm.kh = pl.kh;
    prm.rv = pl.rv;
    const VjpSmem m = vjp_smem(prm.k_pad, prm.kh, prm.rv);
    if (m.stages < 2) return GP_ERR_UNSUPPORTED;
    prm.stages = m.stages;
    prm.sm = m;
    prm.N_pad = pl.N_pad;
    prm.part = part;
    prm.hk = hk;
    prm.err = ctx->dev_err;
    prm.limit_ns = kWaitLimitNs;
    cudaError_t e = cudaErrorInvalidValue;
#define GPK_VJP_CASE(K)                                                                                   \
    case K: {                                                                                             \
        auto fn = kvjp_tc_kernel<K>;                                                                      \
        e = allow_smem(fn, kMaxSmemBytes - 512);                                                          \
        if (e == cudaSuccess) {                                                                           \
            fn<<<pl.grid, kThreads, m.total, s>>>(op.tmA, op.tmB, tmUW, tmWU, tmXt, prm);                  \
            e = cudaGetLastError();                                                                       \
        }                                                                                                 \
        break;                                                                                            \
    }
    prof_begin(ctx, s);
    switch (hyp->kernel) {
        GPK_VJP_CASE(GP_KERNEL_RBF)
        GPK_VJP_CASE(GP_KERNEL_MATERN32)
        GPK_VJP_CASE(GP_KERNEL_MATERN52)
        default: return GP_ERR_UNSUPPORTED;
    }
#undef GPK_VJP_CASE
    prof_end(ctx, s);
    ctx->launches++;
    if (e != cudaSuccess) return GP_ERR_CUDA;

    ScaleVec tl;
    for (int k = 0; k < 64; ++k) tl.v[k] = k < d ? (float)(2.0 / (double)hyp->lengthscale[k]) : 0.0f;
    const float a2kp = (float)hyp->outputscale * kprime_max(hyp->kernel);
    vjp_finish_kernel<<<(unsigned)pl.nblk_f, 256, 0, s>>>(part, pl.n_split, pl.rv, pl.N_pad, xs, Vb, N, d, tl, a2kp,
                                                          scales, pl.rp, gX_dev, lpart);
    // sums[0, d): lengthscale sums, sums[32]: sum H k, sums[33]: sum_c u_c^T w_c
    sum_rows_kernel<<<d, 32, 0, s>>>(lpart, pl.nblk_f, 32, sums);
    sum_rows_kernel<<<1, 32, 0, s>>>(hk, pl.grid, 1, sums + 32);
    coldot2_kernel<<<dim3(kDotBlocks, R), 256, 0, s>>>(U, W, N, dots);
    sum_rows_kernel<<<1, 32, 0, s>>>(dots, R * kDotBlocks, 1, sums + 33);
    ctx->launches += 5;
    if (cudaGetLastError() != cudaSuccess) return GP_ERR_CUDA;
    // small read-back through the context's pinned scratch (4 KB)
    double* hs = reinterpret_cast<double*>(ctx->host_pinned);
    float* hsc = reinterpret_cast<float*>(hs + 64);
    if (cudaMemcpyAsync(hs, sums, sizeof(double) * 64, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaMemcpyAsync(hsc, scales, sizeof(float) * 64, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return GP_ERR_CUDA;
    const double g = (double)hsc[pl.rp];
    // dq/dl_m = -(2 / l_m) sum_i x^_im D_im (F already applied); dq/da^2 = 1/2 sum H k / g^2
    for (int k = 0; k < d; ++k) grad_theta_host[k] = -2.0 / (double)hyp->lengthscale[k] * hs[k];
    grad_theta_host[d] = 0.5 * hs[32] / (g * g);
    grad_theta_host[d + 1] = hs[33];
    return GP_OK;
}

}  // namespace gpk
