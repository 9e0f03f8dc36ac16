// Warp-specialised state-update (flush) kernel for the delta rule with per-channel decay (KDA) on tcgen05 + TMEM, sm_100a.
//
// Replaying n tokens of S_s = (I - beta_s k_s k_s^T) Diag(g_s) S_{s-1} + beta_s k_s v_s^T (Eq. 1, 3) unrolled over the
// window -- the WY form of Appendix C (Eq. 38-42) applied to the state, with the diagonal decays kept as vectors:
//     G_s   = prod_{m<=s} g_m (per channel),   Dn_s = prod_{m>s} g_m
//     Khat_s = G_s * k_s,   Ktil_s = Dn_s * k_s                  n x K     decayed keys (fp32 values: bf16 hi + lo)
//     A_sj  = sum_i k_s[i] k_j[i] prod_{j<m<=s} g_m[i]  (j < s)  n x n     every product of decays formed by multiplication
//     P     = Khat S_0                                           n x V
//     E     = T (V - P),   T = (I + Bd A)^{-1} Bd                n x V
//     S_new = Diag(G_n) S_0 + Ktil^T E                           K x V
//     [U | o] = S_0^T (G_n * [Omega | q]) + E^T (Ktil [Omega | q])         (Eq. 7 and the exact output of the flush step)
// No quotient of cumulative decays is ever formed (they underflow within a window on real gates).
//
// Tile = one head (K = V = 128), TMEM lane = value column; the state is read once by bulk copies into a ring of
// shared-memory stages; the pass-A group splits the S_0 chunks into bf16 hi + lo and leaves G_n * S_0 in the accumulator
// of Ktil^T E (tcgen05.st); one thread issues every MMA; the pass-B group forms E, writes the accumulator (S_new) back
// and stores the sketch rows; the front group builds the ring-only operands two tiles ahead.  Up to 32 tokens per pass
// (the MMAs over tokens take two k-steps); both key operands and the basis operand are per tile and carry hi + lo
// halves, so the B operand of pass A is a double-buffered per-tile window [Khat (32 rows) | G_n * [Omega | q] (32 rows)].
// The kernel runs one CTA per SM (shared memory) and owns all 512 columns of tensor memory: two 64-column slots
// [P | U0] and two 128-column accumulators for alternating tiles, so pass A of tile k + 1 (issued before the E step of
// tile k) never waits for the write-back of tile k.
//
// Front group, 256 threads, thread = (block of eight tokens, channel pair): reads its columns of the staged key and decay rows
// into registers, forms the running products in packed pairs and writes its rows of Khat / Ktil / G_n * W in the operand layouts,
// four bytes at a time.  The pair sums of A inside a block of eight (28) are per-channel products reduced over the channels by one
// transposing butterfly (per-warp partials summed in a fixed order: results are bitwise reproducible); the 8 x 8 blocks that
// couple them are dot products of rescaled keys (the decay product splits at a block boundary without a quotient), all of it in
// fp32; the 16 x 16 block of tokens 16..31 against 0..15 is an mma.sync product of rescaled keys as bf16 hi + lo.  T_11 and T_22 of
// the two blocks of 16 by forward substitution (one column per thread, one warp each) while six warps form Ktil [Omega | q] with mma.sync.
// The E step (E_1 = T_11 x_1, E_2 = T_22 (x_2 - A_21 E_1), 288 packed multiply-adds per lane) runs on the pass-B group, between the
// write-back of one tile and the next, so that the pass-A group only streams.
//
// What bounds it: the chain of the front group (some 10 k cycles a tile; the state of a tile takes 6.6 k at the rate of a copy),
// most of it instruction supply and latency of eight warps: pair sums and Z rows 2.4 k, coupling 1.2 k, operand rows 1.4 k,
// Ktil W and T 2.3 k.  Flush of 16384 heads, 32 tokens: 1030 us with a channel per thread, blocks of 16 tokens (120 pair sums) and
// 190 KB of code; 775 now (0.53 of a copy's rate; 740 to 850 by box).  Not kept: E of the next tile before the write-back (the accumulator is freed
// late: +60 us), T before the wait for the operand set (+40), the coupling products of a level on one warp with its fragments a
// step ahead (spills: +100).
//
// Domain: KDA, bf16 I/O, K = V = 128, rank <= 16; 1..32 tokens per pass, up to 64 tokens per flush in blocks of 32.
#include <type_traits>
#include "internal.cuh"
#include "lanegroup.cuh"
#include "operand_sets.h"
#include "tc_common.cuh"

namespace sketchssm {

namespace {

using namespace tc;

constexpr int kKThreads = 576;       // pass-A group (4 warps), front group part 1 (4 warps), MMA issue warp, state-load warp, pass-B group (4 warps), front group part 2 (4 warps)
constexpr int kKFront = 256;         // threads of the front group
constexpr int kNT = 32;              // tokens per pass
constexpr int kKStages = 8;          // upper bound on the shared-memory stages of state rows
constexpr int kAS2 = 20;             // row stride (floats) of the two 16 x 16 triangles of A
constexpr uint32_t kZPitch = 272u;   // bytes between the rows of the rescaled keys Z[token][channel]: 256 + 16, so that the 8 rows of an ldmatrix fall in different banks
constexpr uint32_t kZHalf = 32u * kZPitch;   // hi rows, then lo rows, for the boundary at token 16 ...
constexpr uint32_t kZ8 = 2u * kZHalf;        // ... then fp32 rows for those at 8 and 24,
constexpr uint32_t kZ8Pitch = 528u;          // 512 + 16 bytes apart: rows that differ by less than eight fall in different banks
constexpr int kOP = 132;             // floats between the columns of Omega in shared memory [16][128]
// Pass-A window [Khat 32 | G_n * W 32]: 64 rows of 16 bytes per group of 8 channels, the groups 16 bytes further apart than
// they need to be, so that the per-channel threads of a warp (4 groups) store to different banks
constexpr uint32_t kLboW = 64u * 16u + 16u;
// Ktil operand (MN-major: 8 channels x 8 tokens per core matrix): the four token groups of a channel group lie side by
// side and the channel groups 16 bytes further apart than that, so the four channel groups a warp stores to for one
// token fall into different banks
constexpr uint32_t kLboT = 128u, kSboT = 4u * 128u + 16u, kKtHalf = (uint32_t)(kK / 8) * kSboT;
constexpr int kKA2 = 2;              // chunk buffers between the pass-A group and the MMA issue warp
constexpr int kNPk = 32;             // columns of [Omega | q]: Omega in 0..R-1, q at column QA = round_up(R, 8) <= 16

struct KSmem {
    uint32_t a2, e, w, w_stride, w_lo, set, set_stride, set_bt, set_bt_lo, set_vv, set_t1, set_bc, set_gn, stg, stg_g,
        stg_beta, stg_q, mats, om, bars, misc, sst, sst_bytes, total;
};

__host__ __device__ inline KSmem make_ksmem(int stages) {
    KSmem s;
    uint32_t off = 0;
    s.a2 = off; off += (uint32_t)kKA2 * 2u * 128u * 16u * 2u;     // 16-row chunk buffers, hi + lo
    s.e = off; off += 2u * 128u * (uint32_t)kNT * 2u;             // E hi + lo: A operand of Ktil^T E (128 x 32 tokens each)
    // B operand of pass A, per tile and double-buffered: 64 rows [Khat (32) | G_n * [Omega | q] (32)] x 128 channels, hi then lo
    s.w = off; s.w_lo = (uint32_t)(kK / 8) * kLboW; s.w_stride = 2u * s.w_lo; off += 2u * s.w_stride;
    // per-tile operand set, double-buffered: Ktil as B operand of Ktil^T E (MN-major, hi | lo), raw value rows, T,
    // Ktil [Omega | q] hi | lo (B operand of the sketch correction), G_n
    s.set = off;
    s.set_bt = 0u; s.set_bt_lo = kKtHalf; s.set_vv = 2u * kKtHalf; s.set_t1 = s.set_vv + 8192u; s.set_bc = s.set_t1 + 3072u;
    s.set_gn = s.set_bc + 4096u;
    s.set_stride = s.set_gn + 512u;
    off += 2u * s.set_stride;
    // staging of the next tile's raw rows: keys [32][256 B], decays [32][256 B]; beta [L] floats, query row (double-buffered: it is
    // read until the tile is finished).  (Value rows go straight into the set.)  Once a tile's rows are in registers the key / decay
    // area is re-used for the rescaled keys Z.
    s.stg_g = 8192u; s.stg_beta = kZ8 + 32u * kZ8Pitch; s.stg_q = s.stg_beta + 256u;
    s.stg = off; off += s.stg_q + 512u;
    s.mats = off; off += 2u * 16u * kAS2 * 4u + 128u + 8u * 32u * 4u + 4u * 128u * 4u;    // A (beta_s A_sj), beta, partial pair sums, products of the decays of eight tokens
    s.om = off; off += 16u * kOP * 4u;                            // Omega of the current head index, fp32 (zero beyond the rank)
    s.bars = off; off += 512u;
    s.misc = off; off += 128u;
    off = (off + 127u) & ~127u;
    s.sst_bytes = 16u * 128u * 4u;
    s.sst = off; off += (uint32_t)stages * s.sst_bytes;
    s.total = off;
    return s;
}

enum { kPro = 0, kPfull = 2, kTfull = 4, kBufFree = 6, kA2free = 8, kA2rdy = 8 + kKA2, kErdy = 8 + 2 * kKA2,
       kStg = 9 + 2 * kKA2, kStDone = 10 + 2 * kKA2, kFull = 12 + 2 * kKA2, kEmpty = 12 + 2 * kKA2 + kKStages,
       kTfree = 12 + 2 * kKA2 + 2 * kKStages, kVals = 14 + 2 * kKA2 + 2 * kKStages, kNumBars = 16 + 2 * kKA2 + 2 * kKStages };

__device__ __forceinline__ void k_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// named barrier 2 over the 256 threads of the front group, and a group-wide bounded wait: one warp polls, the others
// sleep in the barrier
__device__ __forceinline__ void f_sync() { asm volatile("bar.sync 2, 256;" ::: "memory"); }
__device__ __forceinline__ bool f_wait(int ft, uint64_t* bar, uint32_t phase) {
    bool bad = false;
    if (ft < 32) bad = !mbar_wait_bounded(bar, phase);
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 q, %1, 0;\n\t"
        "bar.red.or.pred p, 2, 256, q;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(r)
        : "r"(bad ? 1u : 0u)
        : "memory");
    return r == 0;
}
__device__ __forceinline__ void k_ldmatrix_x4(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void k_mma_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

}  // namespace

__global__ void __launch_bounds__(kKThreads, 1) update_tc_ws_kda_kernel(const Params p) {
    constexpr int K = kK, V = 128, CH = 16, NCH = K / CH, NP = kNPk;
    extern __shared__ __align__(1024) unsigned char smem[];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int gt = tid & 127;
    const int R = p.R, H = p.H, B = p.B;
    const int QA = (R + 7) & ~7;                          // column of the query
    const int NS = p.stages;
    const int n_ring = p.n_before, n_tot = n_ring + (p.has_token ? 1 : 0);     // 1..32 per pass (the launcher sees to it)
    const int ksteps = n_tot > 16 ? 2 : 1;                // 16-token k-steps of the MMAs that contract over tokens
    const KSmem sm = make_ksmem(NS);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + sm.bars);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + sm.misc);
    unsigned char* sStg = smem + sm.stg;

    constexpr uint32_t tmem_cols = 512u;          // one CTA per SM (shared memory): two slots of 64 columns, two accumulators of 128
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        *reinterpret_cast<volatile int*>(smem + sm.misc + 32) = 0;
        for (int i = 0; i < kNumBars; ++i) {
            // one arrival per warp of a stream group: chunk ready, E ready, stage empty, accumulator halves, pass-B done, slot free
            const bool per_warp = (i >= kA2rdy && i <= kErdy) || i == kStDone || i == kStDone + 1 || (i >= kEmpty && i < kVals) || i == kBufFree || i == kBufFree + 1;
            mbar_init(&bars[i], per_warp ? 4 : 1);
        }
        mbar_fence_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    grid_dep_wait();                 // nothing above reads memory another kernel may write
    grid_dep_launch_dependents();
    const uint32_t tmem_base = *tmem_slot;
    const uint32_t lane_sel = (uint32_t)((warp & 3) * 32) << 16;

    // instruction descriptors: bf16 x bf16 -> fp32, M = 128
    const uint32_t idescT = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((128u >> 3) << 17) | ((128u >> 4) << 24);    // K-major x MN-major, N = 128
    const uint32_t idescU = (1u << 4) | (1u << 7) | (1u << 10) | (((uint32_t)NP >> 3) << 17) | ((128u >> 4) << 24);        // K-major x K-major, N = 32
    const uint32_t idescA = (1u << 4) | (1u << 7) | (1u << 10) | ((64u >> 3) << 17) | ((128u >> 4) << 24);                 // K-major x K-major, N = 64
    // canonical no-swizzle layouts (byte offsets)
    //   K-major : elem(mn, k) at (mn%8)*16 + (mn/8)*128 + (k/8)*LBO + (k%8)*2,  LBO = 16*MN
    //   MN-major: elem(mn, k) at (k%8)*16 + (mn%8)*2 + (mn/8)*128 + (k/8)*2048
    constexpr uint32_t SBO = 128, LBO_M = 2048;
    constexpr uint32_t LBO_W = kLboW;                     // pass-A window: 64 rows (+ 16 bytes of padding)
    constexpr uint32_t LBO_C = (uint32_t)NP * 16u;        // Ktil W: 32 rows

    const int tiles_per_h = B;

    // the CTA's sequence of tile numbers (claimed at run time by the front group) travels through a small ring
    volatile int* seq_ring = reinterpret_cast<volatile int*>(smem + sm.misc + 16);
    volatile int* seq_pub = reinterpret_cast<volatile int*>(smem + sm.misc + 32);
    auto seq_get = [&](int k) -> int {          // -2: the wait ran out
#pragma unroll 1
        for (uint32_t it = 0; it < (1u << 22); ++it) {
            if (*seq_pub > k) {
                __threadfence_block();
                return seq_ring[k & 3];
            }
            if (it > 32) __nanosleep(100);
        }
        return -2;
    };
    auto set_ptr = [&](int b) { return smem + sm.set + (uint32_t)b * sm.set_stride; };
    auto w_ptr = [&](int b) { return smem + sm.w + (uint32_t)b * sm.w_stride; };

    const int j = (warp & 3) * 32 + lane;      // value column = TMEM lane of this thread (both stream groups)

    if (warp < 4) {
        // =========================== pass-A group: S_0 chunks -> operands, and the E step ===========================
        uint32_t phPro = 0, phA = 0, phF = 0;
        int gc = 0, stage = 0;
        bool bad = false;

        uint32_t phTf = 0;
        // pass A of the CTA's tile number kt with operand set b = kt & 1; the Ktil^T E accumulator b still holds tile kt - 2
        // until the pass-B group has read it
        auto pass_a = [&](int b, int kt) {
            const float* sGn = reinterpret_cast<const float*>(set_ptr(b) + sm.set_gn);
#pragma unroll 1
            for (int c = 0; c < NCH; ++c) {
                if (c == 0 && kt >= 2) {
                    bad |= !mbar_wait_bounded(&bars[kTfree + b], (phTf >> b) & 1u);
                    phTf ^= 1u << b;
                    tc_fence_after();
                }
                bad |= !mbar_wait_bounded(&bars[kFull + stage], phF);
                const float* sS = reinterpret_cast<const float*>(smem + sm.sst + (size_t)stage * sm.sst_bytes) + j;
                float s0[CH];
#pragma unroll
                for (int ii = 0; ii < CH; ++ii) s0[ii] = sS[ii * V];
                __syncwarp();
                if (lane == 0) k_arrive(&bars[kEmpty + stage]);
                {   // G_n * S_0 goes into the Ktil^T E accumulator, so that the MMAs leave S_new there
                    float ds[CH];
#pragma unroll
                    for (int i4 = 0; i4 < CH / 4; ++i4) {
                        const float4 g4 = *reinterpret_cast<const float4*>(sGn + c * CH + i4 * 4);
                        ds[i4 * 4 + 0] = g4.x * s0[i4 * 4 + 0];
                        ds[i4 * 4 + 1] = g4.y * s0[i4 * 4 + 1];
                        ds[i4 * 4 + 2] = g4.z * s0[i4 * 4 + 2];
                        ds[i4 * 4 + 3] = g4.w * s0[i4 * 4 + 3];
                    }
                    if (!bad) tmem_st16(tmem_base + 128u + (uint32_t)b * 128u + lane_sel + (uint32_t)(c * CH), ds);
                }
                const int ab = c & (kKA2 - 1);
                if (gc >= kKA2) {     // the chunk buffer was read by the MMAs issued kKA2 chunks ago
                    bad |= !mbar_wait_bounded(&bars[kA2free + ab], (phA >> ab) & 1u);
                    phA ^= 1u << ab;
                }
                unsigned char* a2hi = smem + sm.a2 + (size_t)ab * (2u * 128u * CH * 2u);
                unsigned char* a2lo = a2hi + 128u * CH * 2u;
#pragma unroll
                for (int v8 = 0; v8 < CH / 8; ++v8) {
                    uint32_t ohi[4], olo[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) split_bf16x2(s0[v8 * 8 + 2 * e], s0[v8 * 8 + 2 * e + 1], ohi[e], olo[e]);
                    const uint32_t off = (gt & 7) * 16 + (gt >> 3) * SBO + v8 * LBO_M;
                    *reinterpret_cast<uint4*>(a2hi + off) = make_uint4(ohi[0], ohi[1], ohi[2], ohi[3]);
                    *reinterpret_cast<uint4*>(a2lo + off) = make_uint4(olo[0], olo[1], olo[2], olo[3]);
                }
                proxy_fence();
                bad = __any_sync(0xffffffffu, bad);
                if (lane == 0 && !bad) k_arrive(&bars[kA2rdy + ab]);
                ++gc;
                if (++stage == NS) { stage = 0; phF ^= 1u; }
            }
            tmem_st_wait();            // this warp's G_n * S_0 columns are in tensor memory
            tc_fence_before();
            bad = __any_sync(0xffffffffu, bad);
            if (lane == 0 && !bad) k_arrive(&bars[kStDone + b]);
        };
        auto wait_pro = [&](int b) {
            bad |= !mbar_wait_bounded(&bars[kPro + b], (phPro >> b) & 1u);
            phPro ^= 1u << b;
        };

        // (one call site each, here and in the other roles: the bodies are inlined, and the kernel's code has to stay small)
        for (int k = 0; !bad; ++k) {
            const int raw = seq_get(k);
            if (raw < 0) { bad = raw < -1; break; }
            wait_pro(k & 1);
            pass_a(k & 1, k);
        }
        if (bad && lane == 0) record_fault(p.status, kFaultUpdateWait, 103);
    } else if (warp >= 10 && warp < 14) {
        // =========================== pass-B group: S_new written back, then the sketch rows ===========================
        uint32_t phT = 0, phP = 0, phV = 0;
        bool bad = false;
        // E = T (V - P) with T = (I + Bd A)^{-1} Bd solved in two blocks of 16 tokens -> hi + lo A operand of Ktil^T E
        // (chunk-buffer layout, 32 tokens)
        auto do_e = [&](int b) {
            bad |= !mbar_wait_bounded(&bars[kPfull + b], (phP >> b) & 1u);
            phP ^= 1u << b;
            tc_fence_after();
            const unsigned char* set = set_ptr(b);
            const __nv_bfloat16* sV = reinterpret_cast<const __nv_bfloat16*>(set + sm.set_vv);
            const float* sT1 = reinterpret_cast<const float*>(set + sm.set_t1);
            if (!mbar_wait_bounded(&bars[kVals + b], (phV >> b) & 1u)) bad = true;      // the value rows
            phV ^= 1u << b;
            f32x2 x[kNT / 2];                       // pairs of tokens
            {
                float x0[16], x1[16];
                if (!bad) {
                    tmem_ld16(tmem_base + (uint32_t)b * 64u + lane_sel, x0);
                    tmem_ld16(tmem_base + (uint32_t)b * 64u + 16u + lane_sel, x1);
                } else {
#pragma unroll
                    for (int t = 0; t < 16; ++t) { x0[t] = 0.f; x1[t] = 0.f; }
                }
#pragma unroll
                for (int t = 0; t < 16; t += 2) {
                    x[t / 2] = pack2(__bfloat162float(sV[t * V + j]) - x0[t], __bfloat162float(sV[(t + 1) * V + j]) - x0[t + 1]);
                    x[8 + t / 2] = pack2(__bfloat162float(sV[(16 + t) * V + j]) - x1[t], __bfloat162float(sV[(17 + t) * V + j]) - x1[t + 1]);
                }
            }
            // The 32 x 32 system in two blocks of 16 tokens:  E_1 = T_11 x_1,  E_2 = T_22 (x_2 - A_21 E_1)
            const float* sT11 = sT1;
            const float* sT22 = sT1 + 256;
            const float* sA21 = sT1 + 512;
            // the first 4 n4 columns of a row times 2 n4 pairs
            auto row_dot = [&](const float* row, const f32x2* v, int n4) {
                f32x2 a0 = pack2(0.f, 0.f), a1 = a0;
#pragma unroll
                for (int t4 = 0; t4 < 4; ++t4) {
                    if (t4 < n4) {
                        const ulonglong2 m = *reinterpret_cast<const ulonglong2*>(row + t4 * 4);
                        a0 = fma2(m.x, v[2 * t4], a0);
                        a1 = fma2(m.y, v[2 * t4 + 1], a1);
                    }
                }
                float p, q, r, u;
                unpack2(a0, p, q);
                unpack2(a1, r, u);
                return (p + q) + (r + u);
            };
            float e1[16], e2[16];
            f32x2 e1p[8];
#pragma unroll
            for (int s = 0; s < 16; ++s) e1[s] = row_dot(sT11 + s * 16, x, s / 4 + 1);          // T_11 is lower triangular
#pragma unroll
            for (int s = 0; s < 8; ++s) e1p[s] = pack2(e1[2 * s], e1[2 * s + 1]);
#pragma unroll
            for (int s = 0; s < 8; ++s) {
                float u, v;
                unpack2(x[8 + s], u, v);
                x[8 + s] = pack2(u - row_dot(sA21 + (2 * s) * 16, e1p, 4), v - row_dot(sA21 + (2 * s + 1) * 16, e1p, 4));
            }
#pragma unroll
            for (int s = 0; s < 16; ++s) e2[s] = row_dot(sT22 + s * 16, x + 8, s / 4 + 1);
            unsigned char* ehi = smem + sm.e;
            unsigned char* elo = ehi + 128u * (uint32_t)kNT * 2u;
#pragma unroll
            for (int v8 = 0; v8 < kNT / 8; ++v8) {
                uint32_t ohi[4], olo[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float ea = v8 < 2 ? e1[(v8 & 1) * 8 + 2 * q] : e2[(v8 & 1) * 8 + 2 * q];
                    const float eb = v8 < 2 ? e1[(v8 & 1) * 8 + 2 * q + 1] : e2[(v8 & 1) * 8 + 2 * q + 1];
                    split_bf16x2(ea, eb, ohi[q], olo[q]);
                }
                const uint32_t off = (gt & 7) * 16 + (gt >> 3) * SBO + v8 * LBO_M;
                *reinterpret_cast<uint4*>(ehi + off) = make_uint4(ohi[0], ohi[1], ohi[2], ohi[3]);
                *reinterpret_cast<uint4*>(elo + off) = make_uint4(olo[0], olo[1], olo[2], olo[3]);
            }
            proxy_fence();
            tc_fence_before();
            bad = __any_sync(0xffffffffu, bad);
            if (lane == 0 && !bad) k_arrive(&bars[kErdy]);
        };
        for (int k = 0; !bad; ++k) {
            const int tile = seq_get(k);
            if (tile < 0) { bad = tile < -1; break; }
            const int b = k & 1;
            // the E step: the tile's P is complete once its pass A is, and the E operand buffer is free because Ktil^T E of the
            // tile before has completed (waited for below)
            do_e(b);
            const int h = tile / tiles_per_h, bb = tile - h * tiles_per_h;
            const size_t bh = (size_t)bb * H + h;
            float* So = p.state + bh * (size_t)K * V + j;
            bad |= !mbar_wait_bounded(&bars[kTfull + b], (phT >> b) & 1u);      // Ktil^T E and the sketch correction are complete
            phT ^= 1u << b;
            tc_fence_after();
#pragma unroll 1
            for (int c = 0; c < NCH; ++c) {
                if (!bad) {
                    float t[CH];
                    tmem_ld16(tmem_base + 128u + (uint32_t)b * 128u + lane_sel + (uint32_t)(c * CH), t);
                    if (c == NCH - 1) {      // this warp is done with the accumulator: pass A of tile k + 2 may overwrite it
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) k_arrive(&bars[kTfree + b]);
                    }
#pragma unroll
                    for (int ii = 0; ii < CH; ++ii) So[(size_t)(c * CH + ii) * V] = t[ii];
                }
            }
            bad = __any_sync(0xffffffffu, bad);
            // [U | o] = S_0^T (G_n * W) + E^T (Ktil W) from the tile's slot of tensor memory: [correction 32 | U0 32]
            if (!bad) {
                const uint32_t slot = tmem_base + (uint32_t)b * 64u + lane_sel;
                auto rows = [&](auto bf) {
                    constexpr bool BF = decltype(bf)::value;
                    const size_t base = (bh * R) * (size_t)V + j;
                    for (int g0 = 0; g0 < R; g0 += 16) {
                        float u0[16], cr[16];
                        tmem_ld16(slot + 32u + (uint32_t)g0, u0);
                        tmem_ld16(slot + (uint32_t)g0, cr);
                        if (g0 + 16 <= R) {
#pragma unroll
                            for (int e = 0; e < 16; ++e) store_sketch_as<BF>(p, base + (size_t)(g0 + e) * V, u0[e] + cr[e]);
                        } else {
#pragma unroll
                            for (int e = 0; e < 16; ++e)
                                if (g0 + e < R) store_sketch_as<BF>(p, base + (size_t)(g0 + e) * V, u0[e] + cr[e]);
                        }
                    }
                };
                if (p.write_sketch) {
                    if (p.sketch_bf16) rows(std::true_type{}); else rows(std::false_type{});
                }
                if (p.out != nullptr) {       // exact output: the query column
                    float ou, oc;
                    tmem_ld1x2(slot + 32u + (uint32_t)QA, slot + (uint32_t)QA, ou, oc);
                    const float o = ou + oc;
                    if (p.out_bf16) reinterpret_cast<__nv_bfloat16*>(p.out)[bh * V + j] = __float2bfloat16_rn(o);
                    else reinterpret_cast<float*>(p.out)[bh * V + j] = o;
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) k_arrive(&bars[kBufFree + b]);       // the slot is free for pass A of tile k + 2
            }
        }
        if (bad && lane == 0) record_fault(p.status, kFaultUpdateWait, 111);
    } else if (warp == 8) {
        // =========================== MMA issue warp (one thread) ===========================
        if (lane == 0) {
            uint32_t phR = 0, phE = 0, phBuf = 0, phSt = 0;
            bool bad = false;
            int where = 104;                // which wait gave up (status detail): 141 slot free, 142 chunk ready, 143 E ready, 145 accumulator written
            const uint32_t a2base = smem_u32(smem + sm.a2);
            auto step_e = [&](int k) {          // Ktil^T E onto G_n * S_0 (128 columns) and the sketch correction E^T (Ktil W) over the spent P
                const int b = k & 1;
                if (!mbar_wait_bounded(&bars[kErdy], phE)) { bad = true; where = 143; return; }
                phE ^= 1u;
                // G_n * S_0 is in accumulator b (the pass-A group stored it after the pass-B group had read tile k - 2 from it)
                if (!mbar_wait_bounded(&bars[kStDone + b], (phSt >> b) & 1u)) { bad = true; where = 145; return; }
                phSt ^= 1u << b;
                tc_fence_after();
                const uint32_t tmem_t = tmem_base + 128u + (uint32_t)b * 128u;
                const uint32_t tmem_c = tmem_base + (uint32_t)b * 64u;
                const uint32_t e = smem_u32(smem + sm.e);
                const uint32_t bt = smem_u32(set_ptr(b) + sm.set_bt);
                const uint32_t bc = smem_u32(set_ptr(b) + sm.set_bc);
                for (int kk = 0; kk < ksteps; ++kk) {
                    const uint64_t ehi = make_desc(e + (uint32_t)kk * 2u * LBO_M, LBO_M, SBO);
                    const uint64_t elo = make_desc(e + 128u * (uint32_t)kNT * 2u + (uint32_t)kk * 2u * LBO_M, LBO_M, SBO);
                    const uint64_t bthi = make_desc(bt + (uint32_t)kk * 2u * kLboT, kLboT, kSboT);
                    const uint64_t btlo = make_desc(bt + sm.set_bt_lo + (uint32_t)kk * 2u * kLboT, kLboT, kSboT);
                    const uint64_t bchi = make_desc(bc + (uint32_t)kk * 2u * LBO_C, LBO_C, SBO);
                    const uint64_t bclo = make_desc(bc + 2048u + (uint32_t)kk * 2u * LBO_C, LBO_C, SBO);
                    tc_mma_bf16(tmem_t, ehi, bthi, idescT, 1u);
                    tc_mma_bf16(tmem_t, elo, bthi, idescT, 1u);
                    tc_mma_bf16(tmem_t, ehi, btlo, idescT, 1u);
                    tc_mma_bf16(tmem_c, ehi, bchi, idescU, kk ? 1u : 0u);
                    tc_mma_bf16(tmem_c, elo, bchi, idescU, 1u);
                    tc_mma_bf16(tmem_c, ehi, bclo, idescU, 1u);
                }
                tc_commit(&bars[kTfull + b]);
            };
            // The E step of a tile is issued as soon as its E operand is ready, also in the middle of the next tile's pass A
            // (pend_e: the tile whose E step is still to be issued, or -1).
            int pend_e = -1;
            // [P | U0](b) = S_0^T [Khat^T | G_n * W] chunk by chunk: one 64-row window per tile.  Pass A of tile k + 1 starts before the
            // E step of tile k: the stream of S_0 chunks does not wait for the pass-B group (two accumulators).
            for (int k = 0; !bad; ++k) {
                const int raw = seq_get(k);
                if (raw < -1) { bad = true; break; }
                const int b = k & 1;
                const uint32_t slot = tmem_base + (uint32_t)b * 64u;
                const uint32_t whi0 = smem_u32(w_ptr(b));
                const uint32_t wlo0 = whi0 + sm.w_lo;
                // Steps of the tile: -1 the slot's sketch data of tile k - 2 are stored (k >= 2), 0 .. NCH - 1 its chunks; beside them the
                // E step of the tile before, which is all that is left behind the last tile.
                int c = raw < 0 ? NCH : k >= 2 ? -1 : 0;
#pragma unroll 1
                for (uint32_t it = 0; c < NCH || pend_e >= 0; ++it) {
                    if (it >= (1u << 22)) {
                        bad = true;
                        where = c >= NCH ? 143 : c < 0 ? 141 : 142;
                        break;
                    }
                    if (c < NCH) {
                        const int ab = c & (kKA2 - 1);
                        if (mbar_test_wait(c < 0 ? &bars[kBufFree + b] : &bars[kA2rdy + ab], (c < 0 ? phBuf >> b : phR >> ab) & 1u)) {
                            tc_fence_after();
                            it = 0;
                            if (c < 0) {
                                phBuf ^= 1u << b;
                            } else {
                                phR ^= 1u << ab;
                                const uint32_t a2 = a2base + (uint32_t)ab * (2u * 128u * CH * 2u);
                                const uint64_t ahi = make_desc(a2, LBO_M, SBO);
                                const uint64_t alo = make_desc(a2 + 128u * CH * 2u, LBO_M, SBO);
                                const uint64_t whi = make_desc(whi0 + (uint32_t)(c * (CH / 8)) * LBO_W, LBO_W, SBO);
                                const uint64_t wlo = make_desc(wlo0 + (uint32_t)(c * (CH / 8)) * LBO_W, LBO_W, SBO);
                                tc_mma_bf16(slot, ahi, whi, idescA, c ? 1u : 0u);
                                tc_mma_bf16(slot, alo, whi, idescA, 1u);
                                tc_mma_bf16(slot, ahi, wlo, idescA, 1u);
                                tc_commit(&bars[kA2free + ab]);
                                if (c == NCH - 1) tc_commit(&bars[kPfull + b]);
                            }
                            ++c;
                        }
                    }
                    if (pend_e >= 0 && mbar_test_wait(&bars[kErdy], phE)) {
                        step_e(pend_e);
                        pend_e = -1;
                        it = 0;
                        if (bad) break;
                    }
                }
                if (bad || raw < 0) break;
                pend_e = k;
            }
            if (bad) record_fault(p.status, kFaultUpdateWait, where);
        }
    } else if (warp == 9) {
        // =========================== state-load warp: keeps the ring of S_0 stages full ===========================
        int stage = 0, round = 0;
        bool bad = false;
        auto load_tile = [&](int tile) {
            const int h = tile / tiles_per_h, bb = tile - h * tiles_per_h;
            const float* src = p.state + ((size_t)bb * H + h) * (size_t)K * V;
            if (lane == 0)          // (two stages do not cover the latency of memory)
                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(K * V * 4) : "memory");
            for (int c = 0; c < NCH; ++c) {
                if (round > 0) {     // the stage was released by all four stream warps
                    if (!mbar_wait_bounded(&bars[kEmpty + stage], (uint32_t)(round - 1) & 1u)) { bad = true; return; }
                }
                uint64_t* bar = &bars[kFull + stage];
                if (lane == 0) {
                    mbar_expect_tx(bar, sm.sst_bytes);
                    bulk_g2s(smem + sm.sst + (size_t)stage * sm.sst_bytes, src + (size_t)c * CH * V, (uint32_t)(CH * V * 4), bar);
                }
                if (++stage == NS) { stage = 0; ++round; }
            }
        };
        for (int k = 0; !bad; ++k) {
            const int raw = seq_get(k);
            if (raw < 0) { bad = raw < -1; break; }
            load_tile(raw);
        }
        if (bad && lane == 0) record_fault(p.status, kFaultUpdateWait, 107);
    } else {
        // =========================== front group: ring-only operands, tile claiming ===========================
        // 256 threads: thread = (block tb of eight tokens, channel pair cp): its threads build that block's triangle of A, its rows of
        // Khat / Ktil and its rescaled keys.
        const int ft = warp < 8 ? tid - 128 : tid - (kKThreads - 128) + 128;      // 0..255 (warps 4-7, then the last four warps)
        const int tb = ft >> 6;               // token block: tokens 8 tb .. 8 tb + 7 of the pass
        const int cp = ft & 63;               // channels 2 cp, 2 cp + 1
        const int fw = ft >> 5;               // warp of the group, 0..7
        uint32_t phS = 0;
        int filled = 0;                       // tiles whose value rows were requested
        bool dead = false;
        float* sA = reinterpret_cast<float*>(smem + sm.mats);
        float* sBeta = sA + 2 * 16 * kAS2;
        float* sPart = sBeta + kNT;           // [8 warps][32] pair sums over a warp's 64 channels
        float* sProd = sPart + 8 * 32;        // [4 blocks][128 channels] product of a block's decays
        float* sOm = reinterpret_cast<float*>(smem + sm.om);
        int cur_h = -1;

        // ---- tile claiming (thread 0 of the group): per-head-index counters behind the status words ----
        int* sched = p.status + kStatusInts;
        int* cnt = sched + 4;
        int h_claim = (int)(((long long)blockIdx.x * H) / gridDim.x);
        int t_raw = 0;
        auto claim_issue = [&]() { t_raw = atomicAdd(&cnt[h_claim], 1); };
        auto claim_resolve = [&]() -> int {
            for (int attempt = 0; attempt <= H; ++attempt) {
                if (t_raw < tiles_per_h) return h_claim * tiles_per_h + t_raw;
                int best = -1, best_c = tiles_per_h;
                for (int ii = 1; ii <= H; ++ii) {
                    int hh = h_claim + ii;
                    if (hh >= H) hh -= H;
                    const int c = *reinterpret_cast<volatile int*>(&cnt[hh]);
                    if (c < best_c) { best_c = c; best = hh; }
                }
                if (best < 0) return -1;
                h_claim = best;
                t_raw = atomicAdd(&cnt[h_claim], 1);
            }
            return -1;
        };
        auto publish = [&](int k, int tile) {
            seq_ring[k & 3] = tile;
            __threadfence_block();
            *seq_pub = k + 1;
        };

        // One bulk copy per thread from per-thread constants, spread over the first four warps of the group: copy number c
        // belongs to lane c / 4 of warp c % 4.  0..3: ring keys, decays, values, gates; 4..7: the token's key, decay, value, the query.
        const uint32_t stg_beta_bytes = n_ring > 0 ? (uint32_t)(p.L * 4) : 0u;
        const uint32_t stg_bytes = (uint32_t)n_ring * 512u + stg_beta_bytes + (p.has_token ? 512u : 0u) + (p.q != nullptr ? 256u : 0u);
        const int cp_c = (ft < 128 && (ft & 31) < 2) ? (ft & 31) * 4 + (ft >> 5) : 32;
        const unsigned char* cp_base = nullptr;
        size_t cp_stride = 0;
        uint32_t cp_dst = 0, cp_bytes = 0;
        switch (cp_c) {
            case 0: cp_base = p.ring + (size_t)p.tok_base * 256u; cp_stride = p.rl.head_bytes; cp_dst = 0u; cp_bytes = (uint32_t)n_ring * 256u; break;
            case 1: cp_base = p.ring + p.rl.decay_off + (size_t)p.tok_base * 256u; cp_stride = p.rl.head_bytes; cp_dst = sm.stg_g; cp_bytes = (uint32_t)n_ring * 256u; break;
            case 2: cp_base = p.ring + p.rl.v_off + (size_t)p.tok_base * 256u; cp_stride = p.rl.head_bytes; cp_dst = sm.set_vv; cp_bytes = (uint32_t)n_ring * 256u; break;
            case 3: cp_base = p.ring + p.rl.beta_off; cp_stride = p.rl.head_bytes; cp_dst = sm.stg_beta; cp_bytes = stg_beta_bytes; break;
            case 4: cp_base = reinterpret_cast<const unsigned char*>(p.k); cp_stride = (size_t)K * 2; cp_dst = (uint32_t)n_ring * 256u; cp_bytes = p.has_token ? 256u : 0u; break;
            case 5: cp_base = reinterpret_cast<const unsigned char*>(p.decay); cp_stride = (size_t)K * 2; cp_dst = sm.stg_g + (uint32_t)n_ring * 256u; cp_bytes = p.has_token ? 256u : 0u; break;
            case 6: cp_base = reinterpret_cast<const unsigned char*>(p.v); cp_stride = (size_t)V * 2; cp_dst = sm.set_vv + (uint32_t)n_ring * 256u; cp_bytes = p.has_token ? 256u : 0u; break;
            case 7: cp_base = reinterpret_cast<const unsigned char*>(p.q); cp_stride = (size_t)K * 2; cp_dst = sm.stg_q; cp_bytes = p.q != nullptr ? 256u : 0u; break;
            default: break;
        }
        const bool cp_val = cp_c == 2 || cp_c == 6;
        auto stage_tile = [&](int tile, int kt) {       // whole group: keys, decays, gates and the query of tile number kt
            const int h = tile / tiles_per_h, bb = tile - h * tiles_per_h;
            const size_t bw = (size_t)bb * H + h;
            if (ft == 0) mbar_expect_tx(&bars[kStg], stg_bytes);      // (the phase cannot complete before this arrival, whatever the order of the copies)
            __syncwarp();
            if (cp_bytes && !cp_val) bulk_g2s(sStg + cp_dst + (cp_c == 7 ? 256u * (uint32_t)(kt & 1) : 0u), cp_base + bw * cp_stride, cp_bytes, &bars[kStg]);
        };
        auto stage_values = [&](size_t bw, int b) {     // whole group: value rows into the operand set (rows behind the last token stay zero)
            if (ft == 0) mbar_expect_tx(&bars[kVals + b], (uint32_t)n_tot * 256u);
            __syncwarp();
            if (cp_bytes && cp_val) bulk_g2s(set_ptr(b) + cp_dst, cp_base + bw * cp_stride, cp_bytes, &bars[kVals + b]);
        };
        auto next_tile = [&](int k) {          // whole group
            if (ft == 0) {
                const int nxt = claim_resolve();
                publish(k, nxt);
                if (nxt >= 0) claim_issue();
            }
            f_sync();                          // the published entry is the hand-off to the other threads
            const int nxt = seq_ring[k & 3];
            if (nxt >= 0) stage_tile(nxt, k);
        };
        // operand rows that no tile overwrites hold zeros: the padding columns of [Omega | q] in both windows, and the
        // padding columns of Ktil W in both sets; so do the value rows behind the last token
        for (uint32_t o = (uint32_t)ft * 16u; o < 2u * sm.w_stride; o += kKFront * 16u)
            *reinterpret_cast<uint4*>(smem + sm.w + o) = make_uint4(0, 0, 0, 0);
        for (int sb = 0; sb < 2; ++sb)
            for (uint32_t o = (uint32_t)ft * 16u; o < 8192u; o += kKFront * 16u) {
                *reinterpret_cast<uint4*>(set_ptr(sb) + sm.set_vv + o) = make_uint4(0, 0, 0, 0);
                if (o < 4096u) *reinterpret_cast<uint4*>(set_ptr(sb) + sm.set_bc + o) = make_uint4(0, 0, 0, 0);
            }
        proxy_fence();
        f_sync();

        if (ft == 0) claim_issue();
        next_tile(0);
        for (int k = 0; !dead; ++k) {
            const int raw_tile = seq_get(k);
            if (raw_tile < 0) {
                if (raw_tile < -1) {
                    if (ft == 0) record_fault(p.status, kFaultUpdateWait, 108);
                    dead = true;
                }
                break;
            }
            const int tile = raw_tile;
            const int b = k & 1;
            const int h = tile / tiles_per_h, bb = tile - h * tiles_per_h;
            const size_t bh = (size_t)bb * H + h;
            unsigned char* set = set_ptr(b);
            unsigned char* wb = w_ptr(b);

            // gate of the current token: requested early
            float tok_beta = 0.f;
            if (ft < kNT && p.has_token) tok_beta = p.beta[bh];
            // Omega of this head index in shared memory (global loads here would sit on the group's critical path)
            if (h != cur_h) {
                const float* omg = p.omega + (size_t)h * K * R;
                for (int idx = ft; idx < K * 16; idx += kKFront) {
                    const int kk2 = idx >> 4, g = idx & 15;
                    sOm[g * kOP + kk2] = (g < R && p.write_sketch) ? __ldg(omg + (size_t)kk2 * R + g) : 0.f;
                }
                cur_h = h;            // (visible to the group after the barrier below)
            }
            // the staged rows, gates and query row of this tile must have landed
            if (!f_wait(ft, &bars[kStg], phS)) {
                if (ft == 0) record_fault(p.status, kFaultUpdateWait, 106);
                dead = true;
                break;
            }
            phS ^= 1;

            // ---- this thread's channel pair of its block's eight key and decay rows into registers (raw bfloat16 pairs), the
            // product of the block's decays for the other blocks; gates ----
            const int t0 = 8 * tb;
            uint32_t kw[8], gw[8];
#pragma unroll
            for (int s = 0; s < 8; ++s) {
                const bool on = t0 + s < n_tot;
                kw[s] = on ? *reinterpret_cast<const uint32_t*>(sStg + (uint32_t)(t0 + s) * 256u + 4u * (uint32_t)cp) : 0u;
                gw[s] = on ? *reinterpret_cast<const uint32_t*>(sStg + sm.stg_g + (uint32_t)(t0 + s) * 256u + 4u * (uint32_t)cp) : 0x3f803f80u;
            }
            auto pair_of = [](uint32_t w) { return pack2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u)); };
            f32x2 own = pair_of(gw[0]);
#pragma unroll
            for (int s = 1; s < 8; ++s) own = mul2(own, pair_of(gw[s]));
            *reinterpret_cast<f32x2*>(sProd + tb * 128 + 2 * cp) = own;
            const uint32_t qw = p.q != nullptr ? *reinterpret_cast<const uint32_t*>(sStg + sm.stg_q + 256u * (uint32_t)b + 4u * (uint32_t)cp) : 0u;
            if (ft < kNT) {
                const int s = ft;
                float bt = 0.f;
                if (s < n_ring) bt = reinterpret_cast<const float*>(sStg + sm.stg_beta)[p.tok_base + s];
                else if (s < n_tot) bt = tok_beta;
                sBeta[s] = bt;
            }
            f_sync();                  // every thread holds its columns: the key / decay rows of the staging area are free

            f32x2 blk[4];              // products of the decays of all blocks
#pragma unroll
            for (int u = 0; u < 4; ++u) blk[u] = *reinterpret_cast<const f32x2*>(sProd + u * 128 + 2 * cp);
            const f32x2 one2 = pack2(1.f, 1.f);
            const f32x2 g_before = tb == 0 ? one2 : tb == 1 ? blk[0] : tb == 2 ? mul2(blk[0], blk[1]) : mul2(mul2(blk[0], blk[1]), blk[2]);
            const f32x2 g_after = tb == 3 ? one2 : tb == 2 ? blk[3] : tb == 1 ? mul2(blk[2], blk[3]) : mul2(blk[1], mul2(blk[2], blk[3]));
            const f32x2 g_all = mul2(mul2(blk[0], blk[1]), mul2(blk[2], blk[3]));

            auto put2 = [](unsigned char* hi, unsigned char* lo, f32x2 x) {       // a pair as bf16 hi + lo
                float a, c;
                unpack2(x, a, c);
                split_bf16x2(a, c, *reinterpret_cast<uint32_t*>(hi), *reinterpret_cast<uint32_t*>(lo));
            };
            // ---- A_sj = sum_i k_s[i] k_j[i] prod_{j<m<=s} g_m[i].  Inside a block of eight tokens: 28 pair sums as per-channel
            // products, reduced over the warp's 64 channels by a transposing butterfly.  Between blocks the decay product splits at a
            // block boundary without a quotient: X_s = k_s prod_{boundary<=m<=s} g_m against Y_j = k_j prod_{j<m<boundary} g_m, for the
            // boundary at 16 as bf16 hi + lo rows Z[token][channel], for those at 8 and 24 as fp32 rows: inside 16 tokens A is a sum of
            // fp32 products.  (As hi + lo rows and mma.sync products A lost bits there that keys of few large channels show: 2-norm error
            // of S_new after 12 tokens of one channel 2.4e-5 instead of 1.9e-5, of two 1.29e-5 instead of 1.15e-5.  No faster: window of
            // 16384 heads, 32 tokens, 2854 us with those, 2863 with these, runs 0.3 % apart.) ----
            {
                f32x2 k2[8], g2[8];
#pragma unroll
                for (int s = 0; s < 8; ++s) { k2[s] = pair_of(kw[s]); g2[s] = pair_of(gw[s]); }
                float vals[32];
#pragma unroll
                for (int s = 1; s < 8; ++s) {
                    f32x2 r = k2[s];
#pragma unroll
                    for (int jj = 6; jj >= 0; --jj) {
                        if (jj < s) {
                            r = mul2(r, g2[jj + 1]);
                            float a, c;
                            unpack2(mul2(r, k2[jj]), a, c);
                            vals[s * (s - 1) / 2 + jj] = a + c;
                        }
                    }
                }
#pragma unroll
                for (int e = 28; e < 32; ++e) vals[e] = 0.f;
                group_reduce_transpose<32, 32>(vals, lane);      // lane l now holds pair l
                sPart[fw * 32 + lane] = vals[0];

                unsigned char* z16 = sStg + (uint32_t)t0 * kZPitch + 4u * (uint32_t)cp;
                unsigned char* z8 = sStg + kZ8 + (uint32_t)t0 * kZ8Pitch + 8u * (uint32_t)cp;
                // (blocks 0, 1 lie before the boundary at 16 and take Y there, blocks 2, 3 take X; blocks 0, 2 take Y at 8 / 24)
                const f32x2 s16 = tb == 0 ? blk[1] : tb == 3 ? blk[2] : one2;
                if (tb != 0) {
                    f32x2 r = one2;
#pragma unroll
                    for (int s = 0; s < 8; ++s) {
                        r = mul2(r, g2[s]);
                        const f32x2 x = mul2(r, k2[s]);
                        if (tb >= 2) put2(z16 + s * kZPitch, z16 + kZHalf + s * kZPitch, mul2(s16, x));
                        if (tb & 1) *reinterpret_cast<f32x2*>(z8 + s * kZ8Pitch) = x;
                    }
                }
                if (tb != 3) {
                    f32x2 r = one2;
#pragma unroll
                    for (int s = 7; s >= 0; --s) {
                        const f32x2 y = mul2(r, k2[s]);
                        r = mul2(r, g2[s]);
                        if (tb < 2) put2(z16 + s * kZPitch, z16 + kZHalf + s * kZPitch, mul2(s16, y));
                        if (!(tb & 1)) *reinterpret_cast<f32x2*>(z8 + s * kZ8Pitch) = y;
                    }
                }
            }
            f_sync();                  // partial pair sums and Z rows are complete

            float cross[4] = {0.f, 0.f, 0.f, 0.f};
            if (fw >= 6) {
                // ---- A_21 = X Y^T (tokens 16..31 against 0..7, 8..15) as mma.sync products of the Z rows, hi * hi + lo * hi + hi * lo, 16 x 8
                // per warp, kept in registers until the operand set is free.  One warp per scheduler (with those of the 8 x 8 blocks): a
                // step waits for its fragments and for the accumulators of the step before ----
                const uint32_t zb = smem_u32(sStg);
                const uint32_t arow = 16u + (uint32_t)(lane & 15);
                const uint32_t brow = (uint32_t)(lane & 7) + (uint32_t)(fw & 1) * 8u;
                const uint32_t abase = zb + arow * kZPitch + (uint32_t)(lane >> 4) * 16u;
                const uint32_t bbase = zb + brow * kZPitch + (uint32_t)((lane >> 3) & 1) * 16u + (uint32_t)(lane >> 4) * kZHalf;     // hi, then lo
                float c1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 2
                for (int ks = 0; ks < K / 16; ++ks) {
                    uint32_t ahi[4], alo[4], y[4];
                    k_ldmatrix_x4(abase + ks * 32, ahi);
                    k_ldmatrix_x4(bbase + ks * 32, y);
                    k_ldmatrix_x4(abase + kZHalf + ks * 32, alo);
                    k_mma_16816(cross, ahi, y[0], y[1]);
                    k_mma_16816(c1, ahi, y[2], y[3]);
                    k_mma_16816(c1, alo, y[0], y[1]);
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) cross[e] += c1[e];
            } else if (fw >= 2) {
                // ---- the 8 x 8 blocks of tokens t1 .. t1 + 7 against the eight before them (t1 = 8, 24), half of the columns per warp: a lane
                // takes rows u, u + 4, columns w, w + 2 and a quarter of the channels ----
                const int t1 = 8 + 16 * (fw & 1), u = (lane >> 1) & 3, w = (fw >= 4 ? 4 : 0) + (lane & 1);
                const unsigned char* zx = sStg + kZ8 + (uint32_t)(t1 + u) * kZ8Pitch + (uint32_t)(lane >> 3) * 128u;
                const unsigned char* zy = sStg + kZ8 + (uint32_t)(t1 - 8 + w) * kZ8Pitch + (uint32_t)(lane >> 3) * 128u;
                f32x2 acc[2][2];
#pragma unroll
                for (int a = 0; a < 2; ++a)
#pragma unroll
                    for (int c = 0; c < 2; ++c) acc[a][c] = pack2(0.f, 0.f);
#pragma unroll 4
                for (int i = 0; i < K / 4; i += 4) {
                    ulonglong2 x[2], y[2];
#pragma unroll
                    for (int a = 0; a < 2; ++a) {
                        x[a] = *reinterpret_cast<const ulonglong2*>(zx + 4 * a * kZ8Pitch + 4 * i);
                        y[a] = *reinterpret_cast<const ulonglong2*>(zy + 2 * a * kZ8Pitch + 4 * i);
                    }
#pragma unroll
                    for (int a = 0; a < 2; ++a)
#pragma unroll
                        for (int c = 0; c < 2; ++c) acc[a][c] = fma2(x[a].y, y[c].y, fma2(x[a].x, y[c].x, acc[a][c]));
                }
#pragma unroll
                for (int a = 0; a < 2; ++a)
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        float lo, hi;
                        unpack2(acc[a][c], lo, hi);
                        lo += hi;
                        lo += __shfl_xor_sync(0xffffffffu, lo, 8);
                        lo += __shfl_xor_sync(0xffffffffu, lo, 16);
                        const int r0 = t1 + u + 4 * a;
                        if (lane < 8) sA[r0 * kAS2 + w + 2 * c] = sBeta[r0] * lo;
                    }
            } else {
                // ---- beta_s A_sj of the pairs inside the blocks of eight, two blocks per warp (only entries below the diagonal are read) ----
                int s = 1;
                while (s < 8 && (s + 1) * s / 2 <= lane) ++s;        // the pair's later token
                if (lane < 28) {
                    const int jj = lane - s * (s - 1) / 2;
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const int s32 = 16 * fw + 8 * u + s;
                        sA[s32 * kAS2 + 8 * u + jj] = sBeta[s32] * (sPart[(4 * fw + 2 * u) * 32 + lane] + sPart[(4 * fw + 2 * u + 1) * 32 + lane]);
                    }
                }
            }
            proxy_fence();             // (the next tile's rows come in by bulk copies over Z)
            next_tile(k + 1);          // (its barrier:) A is complete and Z has been read: the next tile's rows may come in

            // Up to here nothing of the operand set and window b was touched: they are free once Ktil^T E of tile k - 2 has
            // completed, so everything above overlaps the tail of that tile.
            if (k >= 2) {
                if (!f_wait(ft, &bars[kTfull + b], (uint32_t)((k - 2) >> 1) & 1u)) {
                    if (ft == 0) record_fault(p.status, kFaultUpdateWait, 109);
                    dead = true;
                    break;
                }
            }
            stage_values(bh, b);
            ++filled;
            // ---- running products of this block.  Khat -> window rows 0..31; Ktil -> set (MN-major); G_n * W -> window rows 32.. ----
            {
                unsigned char* wcol = wb + (uint32_t)(cp >> 2) * LBO_W + (uint32_t)(cp & 3) * 4u;              // K-major: k = channel
                unsigned char* bcol = set + sm.set_bt + (uint32_t)(cp & 3) * 4u + (uint32_t)(cp >> 2) * kSboT;   // MN-major: mn = channel
                unsigned char* wrow = wcol + (uint32_t)tb * SBO;
                unsigned char* brow = bcol + (uint32_t)tb * kLboT;
                f32x2 G = g_before;
#pragma unroll
                for (int s = 0; s < 8; ++s) {
                    G = mul2(G, pair_of(gw[s]));
                    put2(wrow + s * 16, wrow + sm.w_lo + s * 16, mul2(G, pair_of(kw[s])));
                }
                f32x2 D = g_after;
#pragma unroll
                for (int s = 7; s >= 0; --s) {
                    put2(brow + s * 16, brow + sm.set_bt_lo + s * 16, mul2(D, pair_of(kw[s])));
                    D = mul2(D, pair_of(gw[s]));
                }
                if (tb == 0) *reinterpret_cast<f32x2*>(set + sm.set_gn + 8 * cp) = g_all;
                // G_n * [Omega | q]: block tb takes every fourth sketch column, the last one the query
                if (p.write_sketch) {
                    for (int g = tb; g < R; g += 4) {
                        unsigned char* at = wcol + (uint32_t)(g & 7) * 16u + (uint32_t)((g >> 3) + 4) * SBO;
                        put2(at, at + sm.w_lo, mul2(g_all, *reinterpret_cast<const f32x2*>(sOm + g * kOP + 2 * cp)));
                    }
                }
                if (tb == 3 && p.q != nullptr) {
                    unsigned char* at = wcol + (uint32_t)(QA & 7) * 16u + (uint32_t)((QA >> 3) + 4) * SBO;
                    put2(at, at + sm.w_lo, mul2(g_all, pair_of(qw)));
                }
                if (fw >= 6) {
                    float* sA21 = reinterpret_cast<float*>(set + sm.set_t1) + 512;
                    const int r0 = lane >> 2, c0 = (fw & 1) * 8 + (lane & 3) * 2;
                    sA21[r0 * 16 + c0] = cross[0];
                    sA21[r0 * 16 + c0 + 1] = cross[1];
                    sA21[(r0 + 8) * 16 + c0] = cross[2];
                    sA21[(r0 + 8) * 16 + c0 + 1] = cross[3];
                }
            }
            f_sync();                  // Ktil is complete

            if ((fw & 3) == 0) {
                // ---- T_bb = (I + Bd A_bb)^{-1} Bd of block fw / 4 by forward substitution: one column per thread, in registers ----
                const int blk = fw >> 2;
                if (lane < 16) {
                    const int c = lane;
                    const int nb = min(max(n_tot - 16 * blk, 0), 16);      // tokens of this block
                    const float* sAb = sA + blk * (16 * kAS2);
                    float tcol[16];
#pragma unroll
                    for (int s = 0; s < 16; ++s) {
                        float acc = 0.f;
#pragma unroll
                        for (int j4 = 0; j4 < (s + 3) / 4; ++j4) {
                            const float4 l4 = *reinterpret_cast<const float4*>(sAb + s * kAS2 + j4 * 4);
                            if (j4 * 4 + 0 < s) acc = fmaf(l4.x, tcol[j4 * 4 + 0], acc);
                            if (j4 * 4 + 1 < s) acc = fmaf(l4.y, tcol[j4 * 4 + 1], acc);
                            if (j4 * 4 + 2 < s) acc = fmaf(l4.z, tcol[j4 * 4 + 2], acc);
                            if (j4 * 4 + 3 < s) acc = fmaf(l4.w, tcol[j4 * 4 + 3], acc);
                        }
                        tcol[s] = (s >= nb || s < c || c >= nb) ? 0.f : (s == c ? 1.f : -acc);
                    }
                    const float bc = sBeta[16 * blk + c];
                    float* sT = reinterpret_cast<float*>(set + sm.set_t1) + blk * 256;
#pragma unroll
                    for (int s = 0; s < 16; ++s) sT[s * 16 + c] = tcol[s] * bc;
                }
            } else {
                // ---- Ktil W: 16 tokens (block fw / 4) x 8 columns of [Omega | q] (columns 8 nt .., nt = fw % 4 - 1) as
                // mma.sync products.  A: the Ktil operand just written (its 8 x 8 core matrices are the row-major fragments
                // ldmatrix wants), hi + lo; B: Omega and q from shared memory into fragments, split into hi + lo in registers ----
                const int mt = fw >> 2, nt = (fw & 3) - 1;
                float acc[4] = {0.f, 0.f, 0.f, 0.f}, c1[4] = {0.f, 0.f, 0.f, 0.f}, c2[4] = {0.f, 0.f, 0.f, 0.f};
                const uint32_t btb = smem_u32(set + sm.set_bt);
                const uint32_t a_row = btb + (uint32_t)(2 * mt + ((lane >> 3) & 1)) * kLboT + (uint32_t)(lane >> 4) * kSboT + (uint32_t)(lane & 7) * 16u;
                const __nv_bfloat16* sq = reinterpret_cast<const __nv_bfloat16*>(sStg + sm.stg_q + 256u * (uint32_t)b);
                const int ncol = p.write_sketch ? R : 0;
                const bool has_q = p.q != nullptr;
                const int g = nt * 8 + (lane >> 2);
                const int src = g < ncol ? 0 : (g == QA && has_q) ? 1 : 2;       // Omega column, query, padding
#pragma unroll 2
                for (int ks = 0; ks < K / 16; ++ks) {
                    uint32_t ahi[4], alo[4], bhi[2], blo[2];
                    k_ldmatrix_x4(a_row + (uint32_t)(2 * ks) * kSboT, ahi);
                    k_ldmatrix_x4(a_row + sm.set_bt_lo + (uint32_t)(2 * ks) * kSboT, alo);
                    const int i0 = ks * 16 + (lane & 3) * 2;
                    float2 w0 = make_float2(0.f, 0.f), w1 = w0;
                    if (src == 0) {
                        w0 = *reinterpret_cast<const float2*>(sOm + g * kOP + i0);
                        w1 = *reinterpret_cast<const float2*>(sOm + g * kOP + i0 + 8);
                    } else if (src == 1) {
                        w0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(sq + i0));
                        w1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(sq + i0 + 8));
                    }
                    split_bf16x2(w0.x, w0.y, bhi[0], blo[0]);
                    split_bf16x2(w1.x, w1.y, bhi[1], blo[1]);
                    k_mma_16816(acc, ahi, bhi[0], bhi[1]);
                    k_mma_16816(c1, alo, bhi[0], bhi[1]);
                    k_mma_16816(c2, ahi, blo[0], blo[1]);
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[e] += c1[e] + c2[e];
                __nv_bfloat16* bchi = reinterpret_cast<__nv_bfloat16*>(set + sm.set_bc);
                __nv_bfloat16* bclo = bchi + 1024;
                auto put = [&](int s, int gc, float x) {
                    __nv_bfloat16 hi, lo;
                    split_bf16(x, hi, lo);
                    const uint32_t o2 = ((uint32_t)(gc & 7) * 16u + (uint32_t)(gc >> 3) * SBO + (uint32_t)(s >> 3) * LBO_C + (uint32_t)(s & 7) * 2u) >> 1;
                    bchi[o2] = hi;
                    bclo[o2] = lo;
                };
                const int s0 = 16 * mt + (lane >> 2), g0 = nt * 8 + (lane & 3) * 2;
                put(s0, g0, acc[0]);
                put(s0, g0 + 1, acc[1]);
                put(s0 + 8, g0, acc[2]);
                put(s0 + 8, g0 + 1, acc[3]);
            }
            proxy_fence();         // operand sets and windows are read by MMAs (async proxy)
            f_sync();
            if (ft == 0) k_arrive(&bars[kPro + b]);
        }
        if (dead && ft < 32) {     // copies that may still be in flight get a short, bounded grace period
            mbar_wait_bounded(&bars[kStg], phS, 1u << 14);
            for (int t = first_unfinished(filled); t < filled; ++t) mbar_wait_bounded(&bars[kVals + set_of_tile(t)], parity_of_tile(t), 1u << 12);
        }
        if (ft == 0) {     // scheduler counters back to zero once every CTA is done claiming
            __threadfence();
            if (atomicAdd(&sched[0], 1) == (int)gridDim.x - 1) {
                for (int hh = 0; hh < H; ++hh) cnt[hh] = 0;
                sched[0] = 0;
                __threadfence();
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
    }
}

// One pass of the kernel over all tiles: ring rows tok_base .. tok_base + n_before - 1 (and the current token).
static int launch_kda_pass(Ctx* ctx, const Params& p_in, cudaStream_t stream) {
    const sketchssm_config& c = ctx->cfg;
    Params p = p_in;
    const uint32_t budget = 227u * 1024u;
    const KSmem fixed = make_ksmem(0);
    if (fixed.total + 2u * fixed.sst_bytes > budget) return SKETCHSSM_UNSUPPORTED_SHAPE;
    int stages = (int)((budget - fixed.total) / fixed.sst_bytes);
    if (stages > kKStages) stages = kKStages;
    if (p.stages >= 2 && p.stages < stages) stages = p.stages;
    p.stages = stages;
    const KSmem sm = make_ksmem(stages);
    const long long n_tiles = (long long)c.batch * c.heads;
    long long grid = (long long)ctx->sm_count;
    if (grid > n_tiles) grid = n_tiles;
    auto kern = update_tc_ws_kda_kernel;
    if ((ctx->last_cuda_error = unlock_smem(ctx, kern)) != cudaSuccess) return SKETCHSSM_CUDA_ERROR;
    if ((ctx->last_cuda_error = launch_kernel(kern, dim3((unsigned)grid), dim3(kKThreads), sm.total, stream, p, p.pdl != 0)) != cudaSuccess)
        return SKETCHSSM_CUDA_ERROR;
    return SKETCHSSM_OK;
}

// Returns SKETCHSSM_UNSUPPORTED_SHAPE outside this kernel's domain (the caller then uses another kernel).  A flush of more
// than 32 tokens is replayed in blocks of 32: every block is one pass over the state, and only the last one (which holds
// the current token) writes the sketch and the exact output.
int launch_update_tc_ws_kda(Ctx* ctx, const Params& p_in, cudaStream_t stream) {
    const sketchssm_config& c = ctx->cfg;
    if (c.kind != SKETCHSSM_KDA || c.io_dtype != SKETCHSSM_BF16 || c.dk != kK || c.dv != 128) return SKETCHSSM_UNSUPPORTED_SHAPE;
    if (c.rank > 16) return SKETCHSSM_UNSUPPORTED_SHAPE;
    const int n_tot = p_in.n_before + (p_in.has_token ? 1 : 0);
    if (n_tot < 1 || n_tot > 2 * kNT) return SKETCHSSM_UNSUPPORTED_SHAPE;
    if (ctx->sm_count == 0) {
        int dev = 0, sms = 0;
        if ((ctx->last_cuda_error = cudaGetDevice(&dev)) != cudaSuccess) return SKETCHSSM_CUDA_ERROR;
        if ((ctx->last_cuda_error = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
            return SKETCHSSM_CUDA_ERROR;
        ctx->sm_count = sms;
    }
    const int passes = (n_tot + kNT - 1) / kNT;
    for (int ps = 0; ps < passes; ++ps) {
        Params p = p_in;
        p.tok_base = ps * kNT;
        if (ps + 1 < passes) {          // 32 ring rows, state only
            p.n_before = kNT;
            p.has_token = 0;
            p.q = nullptr;
            p.out = nullptr;
            p.write_sketch = 0;
        } else {
            p.n_before = p_in.n_before - ps * kNT;
        }
        const int rc = launch_kda_pass(ctx, p, stream);
        if (rc != SKETCHSSM_OK) return rc;
    }
    ctx->last_launches = passes;
    return SKETCHSSM_OK;
}

}  // namespace sketchssm
