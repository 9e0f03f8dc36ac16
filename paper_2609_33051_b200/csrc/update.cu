// State-update (flush) kernel of the SketchSSM hot path (sm_100a), CUDA-core version: every configuration, fp32 throughout.
//
// Every V-column of S is an independent K-vector recurrence under all three transitions: the erase dot <k_s, S[:, j]>
// touches one column only.  A CTA owns the whole state of a head and a warp 16 of its columns: eight lanes share four
// columns, K/8 rows each, in registers.  The state is read once, replayed on chip, projected onto Omega for the sketch
// rows U[g, j] = <S[:, j], omega_g> and onto q for the exact output, and written once (Algorithm 1, flush; Eq. 3, Eq. 7).
//
//   Mamba-2, closed form of Eq. 3:   S <- d S + sum_s (beta_s prod_{j>s} a_j) k_s v_s^T
//   delta rule (GDN, KDA), eight tokens at a time, with G_s = prod_{m<=s} g_m, Dn_s = prod_{m>s} g_m (within the eight):
//     P_s = <G_s k_s, S_0>;  e_s = beta_s (v_s - P_s - sum_{j<s} A_sj e_j),  A_sj = sum_i k_s[i] k_j[i] prod_{j<m<=s} g_m[i];
//     S <- G_8 S_0 + sum_s (Dn_s k_s) e_s^T
//   which is the token-by-token recurrence with the eight erase dots taken from the same state: one decay of the state
//   and one reduction over the rows for eight tokens.  No quotient of decay products is formed.
//
// What bounds it: fp32 issue and the shared-memory reads of the key rows (2 n + r + 1 multiply-adds per state element).
// Four columns per lane: a 128-bit read of a key row feeds eight packed multiply-adds.  One column per lane and 64-column
// tiles, as before, read four times as many key rows and multiplied the state by the decay at every token.  Measured:
// mixed step of 512 sequences x 32 heads, GDN 128 x 128, r = L = 16 (1024 heads flush per call on average): 171 -> 112 us
// a call, of which the decode kernel takes 46 (without the stage 124, with 64-column tiles 131); flush of 3072 KDA heads with
// 8 fp32 tokens: 158 -> 97 us.  The multiply-add pipe is busy 45 % of the time (two CTAs of eight warps: 128 registers a
// thread), fp32 issue 44 %.  Few heads and long GDN windows run update_cols.cu (update_cols_better below).
#include "internal.cuh"
#include "lanegroup.cuh"

namespace sketchssm {

constexpr int kParts = 8;               // lanes that share a group of four columns
constexpr int kTok = 8;                 // tokens replayed together
// Tokens whose key rows are in shared memory at a time.  All rows of a long window at once left room for one CTA per SM or
// for no stage; every further chunk costs two block barriers.  Flush of 8192 heads in us, 16 / 32 at a time: KDA (two rows
// per token) V = 64, L = 32 479 / 652; K = V = 64, L = 64 GDN 396 / 422, Mamba-2 196 / 204; GDN V = 80, L = 64, r = 32 1137 /
// 1229; GDN V = 128, L = 32, r = 32 (no stage either way) 1027 / 969; Mamba-2 V = 64, L = 64 415 / 396.  Chosen
// by how many CTAs fit instead, GDN gained up to 20 % where the column kernel is faster still, and Mamba-2 with V <= 80 lost (444
// heads of V = 80, 32 fp32 tokens 25 -> 37 us).
__host__ __device__ constexpr int update_chunk(int kind, int K, int V) {
    return kind == SKETCHSSM_KDA || K == 64 || (kind == SKETCHSSM_GDN && V == 80) ? 16 : 32;
}
constexpr int kPairs = 32;              // pairs (s, j < s) of kTok tokens, padded from 28
constexpr int kScan = 1024;             // sequences whose phases are looked through at a time

// shared-memory row of K floats split into kParts parts, each padded by 4 floats so that the eight
// parts of a warp read from different banks with 128-bit loads
template <int K>
struct PaddedRow {
    static constexpr int RP = K / kParts;
    static constexpr int stride = K + 4 * kParts;
    __host__ __device__ static constexpr int at(int i) { return i + 4 * (i / RP); }
};

struct UpdateSmem {
    uint32_t kh_off, kt_off, g_off, gram_off, a_off, beta_off, pre_off, suf_off, v_off, e_off, q_off, om_off, list_off, bar_off;
    uint32_t st_off, st_k, st_v, st_gate, st_g, st_tq, st_tk, st_tv, st_tg;      // stage (0 bytes without one)
    uint32_t total;
};

// Omega rows are four floats further apart than a key row: the transposing fill writes consecutive ranks, which would
// otherwise all fall into one bank.
template <int K>
__host__ __device__ constexpr int omega_stride() { return PaddedRow<K>::stride + 4; }

template <int K>
__host__ __device__ inline UpdateSmem make_update_smem(int kind, int n_tot, int R, int V, int L, int io, int mixed, int stage) {
    UpdateSmem u;
    const int ntok = n_tot > 0 ? n_tot : 1;                        // in the stage, and the tokens' weights
    const int nchunk = ntok < update_chunk(kind, K, V) ? ntok : update_chunk(kind, K, V);              // key rows, values and pair sums
    const int nb = (nchunk + kTok - 1) / kTok;
    const int R8 = (R + 7) & ~7;
    const bool delta = kind != SKETCHSSM_MAMBA2, kda = kind == SKETCHSSM_KDA;
    const uint32_t row = PaddedRow<K>::stride * 4;
    uint32_t off = 0;
    u.kt_off = off; off += (uint32_t)(nb * kTok) * row;
    u.kh_off = off; off += kda ? (uint32_t)(nb * kTok) * row : 0u;
    u.g_off = off; off += kda ? (uint32_t)nb * row : 0u;
    u.gram_off = off; off += delta ? (uint32_t)(nb * (K / 32) * kPairs * 4) : 0u;
    u.a_off = off; off += delta ? (uint32_t)(nb * kPairs * 4) : 0u;
    u.beta_off = off; off += (uint32_t)(((ntok + kTok - 1) / kTok) * kTok * 4);
    u.pre_off = off; off += (uint32_t)(nb * kTok * 4);
    u.suf_off = off; off += kind == SKETCHSSM_GDN ? (uint32_t)(nb * kTok * 4) : 0u;
    u.v_off = off; off += (uint32_t)(nchunk * V * io);
    u.e_off = off; off += (uint32_t)(V / 16) * (kTok * 16 * 4);
    u.q_off = off; off += row;
    u.om_off = off; off += (uint32_t)(R8 * omega_stride<K>() * 4);
    u.list_off = off; off += mixed ? (uint32_t)((kScan + 32) * 4) : 0u;
    u.bar_off = off; off += 16u;
    off = (off + 127u) & ~127u;
    u.st_off = u.st_k = u.st_v = u.st_gate = u.st_g = u.st_tq = u.st_tk = u.st_tv = u.st_tg = off;
    if (stage) {
        off += (uint32_t)(K * V * 4);
        u.st_k = off; off += (uint32_t)(ntok * K * io);
        u.st_v = off; off += (uint32_t)(ntok * V * io);
        u.st_gate = off; off += (uint32_t)((kda ? 1 : 2) * L * 4);
        u.st_g = off; off += kda ? (uint32_t)(ntok * K * io) : 0u;
        u.st_tq = off; off += (uint32_t)(K * io);
        u.st_tk = off; off += (uint32_t)(K * io);
        u.st_tv = off; off += (uint32_t)(V * io);
        u.st_tg = off; off += kda ? (uint32_t)(K * io) : 0u;
    }
    u.total = off;
    return u;
}

// Dot products of this lane's rows of four columns with four rows of shared memory: vals[4 t + c].
template <int RP>
__device__ __forceinline__ void dot4(const f32x2 (&c2)[4][RP / 2], const float* row, int stride, float* vals) {
    f32x2 acc[4][4];
#pragma unroll
    for (int i4 = 0; i4 < RP / 4; ++i4) {
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const float4 kq = *reinterpret_cast<const float4*>(row + t * stride + 4 * i4);
            const f32x2 k01 = pack2(kq.x, kq.y), k23 = pack2(kq.z, kq.w);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                acc[t][c] = i4 == 0 ? mul2(k01, c2[c][0]) : fma2(k01, c2[c][2 * i4], acc[t][c]);
                acc[t][c] = fma2(k23, c2[c][2 * i4 + 1], acc[t][c]);
            }
        }
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            float a, b;
            unpack2(acc[t][c], a, b);
            vals[4 * t + c] = a + b;
        }
    }
}

// Sums over the eight parts (lane bits 2..4): part p ends up with the four columns of row p in v[0..3].
__device__ __forceinline__ void reduce_parts(float (&v)[32], int lane) {
#pragma unroll
    for (int lvl = 0; lvl < 3; ++lvl) {
        const int o = 16 >> lvl, half = 16 >> lvl;
        const bool upper = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            if (i < half) {
                const float send = upper ? v[i] : v[i + half];
                const float keep = upper ? v[i + half] : v[i];
                v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
        }
    }
}

// Resident CTAs that the register file is divided for: 128 registers a thread hold 64 of the state, the 32 accumulators
// of four dot products and the key rows in flight.
template <int V>
__host__ __device__ constexpr int update_ctas() { return V == 128 ? 2 : V == 80 ? 3 : 4; }

template <int KIND, typename IO, int K, int V>
__global__ void __launch_bounds__(2 * V, update_ctas<V>()) update_kernel(const Params p) {
    constexpr int T = 2 * V;                        // V / 16 warps
    using PR = PaddedRow<K>;
    constexpr int RP = PR::RP, KS = PR::stride, OS = omega_stride<K>();
    constexpr bool DELTA = KIND != SKETCHSSM_MAMBA2, KDA = KIND == SKETCHSSM_KDA;
    constexpr int kChunk = update_chunk(KIND, K, V);
    extern __shared__ __align__(128) unsigned char smem[];

    const int R = p.R, H = p.H, B = p.B;
    const int R8 = (R + 7) & ~7;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int part = lane >> 2;                     // which rows: part * RP ..
    const int j0 = warp * 16 + (lane & 3) * 4;      // first of this lane's four columns
    const bool mixed = p.n_dev != nullptr;

    // With per-sequence phases the flush may run beside the decode kernel that was launched just before it (each leaves
    // the other's sequences alone, and that kernel let its dependents start only after its own predecessor was done), so
    // it waits at its end instead; the launcher asks for it.
    if (!p.late_wait) grid_dep_wait();
    grid_dep_launch_dependents();

    const bool staged = p.stages != 0;
    const UpdateSmem us = make_update_smem<K>(KIND, mixed ? p.n_cap : p.n_before + (p.has_token ? 1 : 0), R, V, p.L,
                                              (int)sizeof(IO), mixed, staged);
    float* sKt = reinterpret_cast<float*>(smem + us.kt_off);
    float* sKh = reinterpret_cast<float*>(smem + us.kh_off);
    float* sG = reinterpret_cast<float*>(smem + us.g_off);
    float* sGram = reinterpret_cast<float*>(smem + us.gram_off);
    float* sA = reinterpret_cast<float*>(smem + us.a_off);
    float* sBeta = reinterpret_cast<float*>(smem + us.beta_off);
    float* sPre = reinterpret_cast<float*>(smem + us.pre_off);      // GDN: decay up to a token of its eight; Mamba-2: [0] the total
    float* sSuf = reinterpret_cast<float*>(smem + us.suf_off);      // GDN: decay behind it
    IO* sV = reinterpret_cast<IO*>(smem + us.v_off);
    float* sE = reinterpret_cast<float*>(smem + us.e_off) + warp * (kTok * 16);
    float* sQ = reinterpret_cast<float*>(smem + us.q_off);
    float* sOm = reinterpret_cast<float*>(smem + us.om_off);
    int* sList = reinterpret_cast<int*>(smem + us.list_off);
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem + us.bar_off);
    float* sTok = reinterpret_cast<float*>(smem + us.bar_off + 8);  // the current token's beta and scalar decay (staged)

    // One head ahead, by bulk copies into a stage: the state, the buffered tokens and the current token's rows.  A CTA holds
    // one head in registers, and two to four CTAs per SM do not cover the latency of memory between two heads by
    // themselves.  The token's scalar gates travel through the registers of the thread that issues the copies.
    int h_staged = -1;                              // head index whose Omega is in shared memory
    uint32_t parity = 0;
    bool failed = false;
    float next_beta = 0.f, next_decay = 1.f;
    auto request = [&](int b, int h, int n_ring) {      // thread 0
        const size_t bh = (size_t)b * H + h;
        const unsigned char* rh = p.ring + bh * p.rl.head_bytes;
        constexpr uint32_t kRow = (uint32_t)(K * sizeof(IO)), vRow = (uint32_t)(V * sizeof(IO));
        const uint32_t gates = (uint32_t)((KDA ? 1 : 2) * p.L * 4);
        uint32_t bytes = (uint32_t)(K * V * 4);
        if (n_ring > 0) bytes += (uint32_t)n_ring * ((KDA ? 2 : 1) * kRow + vRow) + gates;
        if (p.has_token) bytes += (KDA ? 2 : 1) * kRow + vRow;
        if (p.q != nullptr) bytes += kRow;
        mbar_expect_tx(bar, bytes);
        bulk_g2s(smem + us.st_off, p.state + bh * (size_t)(K * V), (uint32_t)(K * V * 4), bar);
        if (n_ring > 0) {
            bulk_g2s(smem + us.st_k, rh, (uint32_t)n_ring * kRow, bar);
            bulk_g2s(smem + us.st_v, rh + p.rl.v_off, (uint32_t)n_ring * vRow, bar);
            bulk_g2s(smem + us.st_gate, rh + p.rl.beta_off, gates, bar);
            if constexpr (KDA) bulk_g2s(smem + us.st_g, rh + p.rl.decay_off, (uint32_t)n_ring * kRow, bar);
        }
        if (p.has_token) {
            bulk_g2s(smem + us.st_tk, reinterpret_cast<const IO*>(p.k) + bh * K, kRow, bar);
            bulk_g2s(smem + us.st_tv, reinterpret_cast<const IO*>(p.v) + bh * V, vRow, bar);
            if constexpr (KDA) bulk_g2s(smem + us.st_tg, reinterpret_cast<const IO*>(p.decay) + bh * K, kRow, bar);
            next_beta = p.beta[bh];
            if constexpr (!KDA) next_decay = reinterpret_cast<const float*>(p.decay)[bh];
        }
        if (p.q != nullptr) bulk_g2s(smem + us.st_tq, reinterpret_cast<const IO*>(p.q) + bh * K, kRow, bar);
    };

    // n_next: ring fill of the CTA's next head (b_next, h_next); negative if there is none
    auto replay = [&](int b, int h, int n_ring, int b_next, int h_next, int n_next) {
        const size_t bh = (size_t)b * H + h;
        const int n_tot = n_ring + (p.has_token ? 1 : 0);

        // ---- state -> registers ----
        float4 raw[RP];
        const unsigned char* rh = p.ring + bh * p.rl.head_bytes;
        const IO* rk = reinterpret_cast<const IO*>(rh);
        const IO* rv = reinterpret_cast<const IO*>(rh + p.rl.v_off);
        const float* rbeta = reinterpret_cast<const float*>(rh + p.rl.beta_off);
        const float* rdec = reinterpret_cast<const float*>(rh + p.rl.decay_off);
        const IO* tk = reinterpret_cast<const IO*>(p.k) + bh * K;
        const IO* tv = reinterpret_cast<const IO*>(p.v) + bh * V;
        const IO* tq = reinterpret_cast<const IO*>(p.q) + bh * K;
        const IO* tg = reinterpret_cast<const IO*>(p.decay) + bh * K;            // KDA
        const float* tbeta = p.beta + bh;
        const float* tdec = reinterpret_cast<const float*>(p.decay) + bh;        // scalar decays
        if (staged) {
            rk = reinterpret_cast<const IO*>(smem + us.st_k);
            rv = reinterpret_cast<const IO*>(smem + us.st_v);
            rbeta = reinterpret_cast<const float*>(smem + us.st_gate);
            rdec = KDA ? reinterpret_cast<const float*>(smem + us.st_g) : rbeta + p.L;
            tk = reinterpret_cast<const IO*>(smem + us.st_tk);
            tv = reinterpret_cast<const IO*>(smem + us.st_tv);
            tq = reinterpret_cast<const IO*>(smem + us.st_tq);
            tg = reinterpret_cast<const IO*>(smem + us.st_tg);
            tbeta = sTok;
            tdec = sTok + 1;
            // (KDA at 128 registers spills 24 to 32 bytes with the wait rolled or in four copies by pragma, none as the compiler has it: sketch of
            // 8192 heads of 128 x 128 177 -> 160 us, flush of four fp32 tokens 344 -> 313; Mamba-2, V = 80 is 5 % faster rolled)
            failed = !mbar_wait_bounded<!KDA>(bar, parity);
            if (failed) mbar_wait_bounded<!KDA>(bar, parity, 1u << 14);    // a last chance for copies in flight before the CTA leaves
            parity ^= 1u;
            const float* Ss = reinterpret_cast<const float*>(smem + us.st_off) + (part * RP) * V + j0;
#pragma unroll
            for (int i = 0; i < RP; ++i) raw[i] = *reinterpret_cast<const float4*>(Ss + i * V);
        } else {
            const float* Sg = p.state + bh * (size_t)(K * V) + (size_t)(part * RP) * V + j0;
#pragma unroll
            for (int i = 0; i < RP; ++i) raw[i] = *reinterpret_cast<const float4*>(Sg + (size_t)i * V);
        }

        f32x2 c2[4][RP / 2];
#pragma unroll
        for (int i = 0; i < RP / 2; ++i) {
            c2[0][i] = pack2(raw[2 * i].x, raw[2 * i + 1].x);
            c2[1][i] = pack2(raw[2 * i].y, raw[2 * i + 1].y);
            c2[2][i] = pack2(raw[2 * i].z, raw[2 * i + 1].z);
            c2[3][i] = pack2(raw[2 * i].w, raw[2 * i + 1].w);
        }
        const int row = part * (RP + 4);            // this lane's rows inside a padded row

        // kChunk tokens at a time: their rows -> shared memory (fp32), then the replay
#pragma unroll 1
        for (int c0 = 0; c0 == 0 || c0 < n_tot; c0 += kChunk) {
            const int n_here = min(n_tot - c0, kChunk), nb = (n_here + kTok - 1) / kTok;
            const bool last = c0 + kChunk >= n_tot;
            if (c0 > 0) __syncthreads();                 // the previous tokens' rows have been read
            if constexpr (DELTA) {
                // a thread per (eight tokens, channel)
                for (int idx = tid; idx < nb * K; idx += T) {
                    const int blk = idx / K, i = idx % K;
                    float k[kTok], g[kTok];
#pragma unroll
                    for (int s = 0; s < kTok; ++s) {
                        const int t = c0 + blk * kTok + s;
                        k[s] = 0.f;
                        g[s] = 1.f;
                        if (t < n_ring) {
                            k[s] = static_cast<float>(rk[(size_t)t * K + i]);
                            g[s] = KDA ? static_cast<float>(reinterpret_cast<const IO*>(rdec)[(size_t)t * K + i]) : rdec[t];
                        } else if (t < n_tot) {
                            k[s] = static_cast<float>(tk[i]);
                            g[s] = KDA ? static_cast<float>(tg[i]) : *tdec;
                        }
                    }
                    const int at = blk * kTok * KS + PR::at(i);
                    float pre = 1.f, suf = 1.f;
                    if constexpr (KDA) {
#pragma unroll
                        for (int s = 0; s < kTok; ++s) {
                            pre *= g[s];
                            sKh[at + s * KS] = pre * k[s];
                        }
                        sG[blk * KS + PR::at(i)] = pre;
#pragma unroll
                        for (int s = kTok - 1; s >= 0; --s) {
                            sKt[at + s * KS] = suf * k[s];
                            suf *= g[s];
                        }
                    } else {
#pragma unroll
                        for (int s = 0; s < kTok; ++s) sKt[at + s * KS] = k[s];
                        if (i == 0) {                // scalar decays are applied to the dot products and the e instead
#pragma unroll
                            for (int s = 0; s < kTok; ++s) {
                                pre *= g[s];
                                sPre[blk * kTok + s] = pre;
                            }
#pragma unroll
                            for (int s = kTok - 1; s >= 0; --s) {
                                sSuf[blk * kTok + s] = suf;
                                suf *= g[s];
                            }
                        }
                    }
                    // this channel's term of every A_sj, summed over the warp's 32 channels: lane l ends up with pair l
                    float w[kTok], pr[kPairs];
#pragma unroll
                    for (int s = 0; s < kTok; ++s) {
#pragma unroll
                        for (int j = 0; j < s; ++j) {
                            w[j] *= g[s];
                            pr[s * (s - 1) / 2 + j] = k[s] * w[j];
                        }
                        w[s] = k[s];
                    }
#pragma unroll
                    for (int i2 = kTok * (kTok - 1) / 2; i2 < kPairs; ++i2) pr[i2] = 0.f;
                    group_reduce_transpose<32, kPairs>(pr, lane);
                    sGram[(blk * (K / 32) + i / 32) * kPairs + lane] = pr[0];
                }
                for (int s = tid; s < nb * kTok; s += T) sBeta[s] = c0 + s < n_ring ? rbeta[c0 + s] : c0 + s < n_tot ? *tbeta : 0.f;
            } else {
                for (int idx = tid; idx < n_here * (K / 4); idx += T) {
                    const int s = idx / (K / 4), i = 4 * (idx % (K / 4));
                    float k[4];
                    ld4(c0 + s < n_ring ? rk + (size_t)(c0 + s) * K + i : tk + i, k);
                    st4(sKt + s * KS + PR::at(i), k);
                }
                // w_s = beta_s prod_{j>s} a_j and the total decay, by a warp scan over up to 64 tokens
                if (warp == 0 && c0 == 0) {
                    float a[2], bt[2];
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const int s = lane + 32 * u;
                        a[u] = s < n_ring ? rdec[s] : s < n_tot ? *tdec : 1.f;
                        bt[u] = s < n_ring ? rbeta[s] : s < n_tot ? *tbeta : 0.f;
                    }
                    float after = 1.f;               // product of the decays behind this half
#pragma unroll
                    for (int u = 1; u >= 0; --u) {
                        float incl = a[u];
#pragma unroll
                        for (int o = 1; o < 32; o <<= 1) {
                            const float other = __shfl_down_sync(0xffffffffu, incl, o);
                            if (lane + o < 32) incl *= other;
                        }
                        float excl = __shfl_down_sync(0xffffffffu, incl, 1);
                        if (lane == 31) excl = 1.f;
                        if (lane + 32 * u < n_tot) sBeta[lane + 32 * u] = bt[u] * (excl * after);
                        after *= __shfl_sync(0xffffffffu, incl, 0);
                    }
                    if (lane == 0) sPre[0] = after;
                }
            }
            {
                constexpr int PV = 16 / (int)sizeof(IO), in_row = V / PV;        // 16-byte units
                const uint4* ring_v = reinterpret_cast<const uint4*>(rv);
                const uint4* tok_v = reinterpret_cast<const uint4*>(tv);
                for (int idx = tid; idx < n_here * in_row; idx += T) {
                    const int at = c0 * in_row + idx;
                    reinterpret_cast<uint4*>(sV)[idx] = at < n_ring * in_row ? ring_v[at] : tok_v[at - n_ring * in_row];
                }
            }
            if (p.q != nullptr && c0 == 0) {
                for (int i = tid; i < K / 4; i += T) {
                    float q[4];
                    ld4(tq + 4 * i, q);
                    st4(sQ + PR::at(4 * i), q);
                }
            }
            if (p.write_sketch && h != h_staged) {
                const float* og = p.omega + (size_t)h * K * R;
#pragma unroll 4
                for (int idx = tid; idx < K * R; idx += T) {
                    const int i = idx / R, g = idx % R;
                    sOm[g * OS + PR::at(i)] = og[idx];
                }
                for (int idx = tid; idx < (R8 - R) * K; idx += T) sOm[(R + idx / K) * OS + PR::at(idx % K)] = 0.f;
                h_staged = h;
            }
            // (every thread's wait on the stage; a CTA that gives up leaves its heads as they are)
            if (__syncthreads_or(failed)) {
                failed = true;
                return;
            }
            if (staged && last && tid == 0 && n_next >= 0) request(b_next, h_next, n_next);
            if constexpr (DELTA) {
                // beta_s A_sj
                for (int idx = tid; idx < nb * kPairs; idx += T) {
                    const int blk = idx / kPairs, pair = idx % kPairs;
                    float a = 0.f;
#pragma unroll
                    for (int c = 0; c < K / 32; ++c) a += sGram[(blk * (K / 32) + c) * kPairs + pair];
                    int s = 1;
                    while (s < kTok && (s + 1) * s / 2 <= pair) ++s;      // the pair's later token
                    sA[idx] = s < kTok ? sBeta[blk * kTok + s] * a : 0.f;
                }
                __syncthreads();
            }

            if constexpr (!DELTA) {
                if (n_tot > 0 && c0 == 0) {
                    const f32x2 d2 = pack2(sPre[0], sPre[0]);
#pragma unroll
                    for (int c = 0; c < 4; ++c)
#pragma unroll
                        for (int i = 0; i < RP / 2; ++i) c2[c][i] = mul2(c2[c][i], d2);
                }
            }
            for (int blk = 0; blk < nb; ++blk) {
                const int s0 = blk * kTok;
                const int nt = min(kTok, n_here - s0);
                const int mine = s0 + part;              // this lane's token where a lane stands for one
                float x[4];
                if constexpr (DELTA) {
                    float vals[32];
                    const float* kh = (KDA ? sKh : sKt) + s0 * KS + row;
                    dot4<RP>(c2, kh, KS, vals);
                    if (nt > 4) {
                        dot4<RP>(c2, kh + 4 * KS, KS, vals + 16);
                    } else {
#pragma unroll
                        for (int i = 16; i < 32; ++i) vals[i] = 0.f;
                    }
                    reduce_parts(vals, lane);
                    float v[4] = {0.f, 0.f, 0.f, 0.f};
                    if (mine < n_here) ld4(sV + mine * V + j0, v);
                    const float bt = sBeta[mine], pre = KIND == SKETCHSSM_GDN ? sPre[mine] : 1.f;
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        x[c] = mine < n_here ? bt * (v[c] - (KIND == SKETCHSSM_GDN ? pre * vals[c] : vals[c])) : 0.f;
                } else {
                    float v[4] = {0.f, 0.f, 0.f, 0.f};
                    if (mine < n_here) ld4(sV + mine * V + j0, v);
                    const float w = mine < n_here ? sBeta[c0 + mine] : 0.f;
#pragma unroll
                    for (int c = 0; c < 4; ++c) x[c] = w * v[c];
                }
                __syncwarp();                            // the previous block's e have been read
                st4(sE + part * 16 + (lane & 3) * 4, x);
                __syncwarp();
                if constexpr (DELTA) {
                    // forward substitution, one column per lane
                    if (lane < 16) {
                        float e[kTok], a[kPairs];
#pragma unroll
                        for (int s = 0; s < kTok; ++s) e[s] = sE[s * 16 + lane];
#pragma unroll
                        for (int i = 0; i < kPairs / 4 - 1; ++i) ld4(sA + blk * kPairs + 4 * i, a + 4 * i);
#pragma unroll
                        for (int j = 0; j < kTok - 1; ++j) {
#pragma unroll
                            for (int s = j + 1; s < kTok; ++s) e[s] = fmaf(-a[s * (s - 1) / 2 + j], e[j], e[s]);
                        }
#pragma unroll
                        for (int s = 0; s < kTok; ++s) sE[s * 16 + lane] = KIND == SKETCHSSM_GDN ? sSuf[s0 + s] * e[s] : e[s];
                    }
                    __syncwarp();
#pragma unroll
                    for (int i4 = 0; i4 < RP / 4; ++i4) {
                        f32x2 g01, g23;
                        if constexpr (KDA) {
                            const float4 g = *reinterpret_cast<const float4*>(sG + blk * KS + row + 4 * i4);
                            g01 = pack2(g.x, g.y);
                            g23 = pack2(g.z, g.w);
                        } else {
                            g01 = g23 = pack2(sPre[s0 + kTok - 1], sPre[s0 + kTok - 1]);
                        }
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            c2[c][2 * i4] = mul2(c2[c][2 * i4], g01);
                            c2[c][2 * i4 + 1] = mul2(c2[c][2 * i4 + 1], g23);
                        }
                    }
                }
                const float* kt = sKt + s0 * KS + row;
#pragma unroll 2
                for (int s = 0; s < nt; ++s) {
                    const float4 e = *reinterpret_cast<const float4*>(sE + s * 16 + (lane & 3) * 4);
                    const f32x2 e2[4] = {pack2(e.x, e.x), pack2(e.y, e.y), pack2(e.z, e.z), pack2(e.w, e.w)};
#pragma unroll
                    for (int i4 = 0; i4 < RP / 4; ++i4) {
                        const float4 kq = *reinterpret_cast<const float4*>(kt + s * KS + 4 * i4);
                        const f32x2 k01 = pack2(kq.x, kq.y), k23 = pack2(kq.z, kq.w);
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            c2[c][2 * i4] = fma2(k01, e2[c], c2[c][2 * i4]);
                            c2[c][2 * i4 + 1] = fma2(k23, e2[c], c2[c][2 * i4 + 1]);
                        }
                    }
                }
            }
        }

        // ---- write the updated state back ----
        if (p.write_state && n_tot > 0) {
            float* So = p.state + bh * (size_t)(K * V) + (size_t)(part * RP) * V + j0;
#pragma unroll
            for (int i = 0; i < RP / 2; ++i) {
                float4 lo, hi;
                unpack2(c2[0][i], lo.x, hi.x);
                unpack2(c2[1][i], lo.y, hi.y);
                unpack2(c2[2][i], lo.z, hi.z);
                unpack2(c2[3][i], lo.w, hi.w);
                *reinterpret_cast<float4*>(So + (size_t)(2 * i) * V) = lo;
                *reinterpret_cast<float4*>(So + (size_t)(2 * i + 1) * V) = hi;
            }
        }

        // ---- exact output o[j] = <S_new[:, j], q> ----
        if (p.out != nullptr) {
            f32x2 acc[4];
#pragma unroll
            for (int i4 = 0; i4 < RP / 4; ++i4) {
                const float4 q = *reinterpret_cast<const float4*>(sQ + row + 4 * i4);
                const f32x2 q01 = pack2(q.x, q.y), q23 = pack2(q.z, q.w);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    acc[c] = i4 == 0 ? mul2(q01, c2[c][0]) : fma2(q01, c2[c][2 * i4], acc[c]);
                    acc[c] = fma2(q23, c2[c][2 * i4 + 1], acc[c]);
                }
            }
            float o[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float lo, hi;
                unpack2(acc[c], lo, hi);
                o[c] = lo + hi;
#pragma unroll
                for (int m = 16; m >= 4; m >>= 1) o[c] += __shfl_xor_sync(0xffffffffu, o[c], m);
            }
            if (part == 0) {
                if (p.out_bf16) st4(reinterpret_cast<__nv_bfloat16*>(p.out) + bh * V + j0, o);
                else st4(reinterpret_cast<float*>(p.out) + bh * V + j0, o);
            }
        }

        // ---- sketch rows U[g, j] = <S_new[:, j], omega_g>, eight ranks at a time ----
        if (p.write_sketch) {
            for (int g0 = 0; g0 < R8; g0 += 8) {
                float vals[32];
                dot4<RP>(c2, sOm + g0 * OS + row, OS, vals);
                dot4<RP>(c2, sOm + (g0 + 4) * OS + row, OS, vals + 16);
                reduce_parts(vals, lane);
                if (g0 + part < R) {
                    const size_t at = (bh * R + g0 + part) * V + j0;
                    if (p.sketch_bf16) st4(reinterpret_cast<__nv_bfloat16*>(p.sketch) + at, vals);
                    else st4(p.sketch + at, vals);
                }
            }
        }
    };

    if (staged) {
        if (tid == 0) {
            mbar_init(bar, 1);
            mbar_fence_init();
        }
        __syncthreads();
    }
    // CTAs are persistent and take contiguous ranges of (head index, sequence) items: Omega is staged once per head index.
    // Lock step: every sequence, at the same ring fill.  Per-sequence phases: the flushing sequences of the batch, kScan
    // entries of the phase array at a time, listed in shared memory (every CTA builds the same list).  A grid of one CTA
    // per head, most of which had nothing to do, spent more time on starting CTAs than on the flush.  (One loop for both:
    // the body is some 40 KB of code, and a second copy of it was measured in instruction-cache misses.)
    int* sCount = sList + kScan;
    for (int base = 0; base < B; base += kScan) {
        int n_seq = B;
        if (mixed) {
            constexpr int kWarps = T / 32, kPer = (kScan / 32 + kWarps - 1) / kWarps;     // rows of 32 sequences per warp
            int cnt = 0;
#pragma unroll
            for (int u = 0; u < kPer; ++u) {
                const int r = warp * kPer + u, b = base + 32 * r + lane;
                cnt += __popc(__ballot_sync(0xffffffffu, r < kScan / 32 && b < B && p.n_dev[b] < 0));
            }
            if (lane == 0) sCount[warp] = cnt;
            __syncthreads();
            int at = 0;
            n_seq = 0;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                const int c = sCount[w];
                if (w < warp) at += c;
                n_seq += c;
            }
            for (int u = 0; u < kPer; ++u) {
                const int r = warp * kPer + u, b = base + 32 * r + lane;
                const bool on = r < kScan / 32 && b < B && p.n_dev[b] < 0;
                const uint32_t bal = __ballot_sync(0xffffffffu, on);
                if (on) sList[at + __popc(bal & ((1u << lane) - 1u))] = b;
                at += __popc(bal);
            }
            __syncthreads();
        }
        const long long items = (long long)n_seq * H;
        const int i0 = (int)(items * blockIdx.x / gridDim.x), i1 = (int)(items * (blockIdx.x + 1) / gridDim.x);
        auto item = [&](int i, int& b, int& h, int& n) {
            h = i / n_seq;
            b = i - h * n_seq;
            n = p.n_before;
            if (mixed) {
                b = sList[b];
                n = -p.n_dev[b] - 1;
            }
        };
        int b = 0, h = 0, n = 0;
        if (i0 < i1) {
            item(i0, b, h, n);
            if (staged && tid == 0) {
                request(b, h, n);
                sTok[0] = next_beta;
                sTok[1] = next_decay;
            }
        }
        __syncthreads();
        for (int i = i0; i < i1; ++i) {
            int b_next = 0, h_next = 0, n_next = -1;
            if (i + 1 < i1) item(i + 1, b_next, h_next, n_next);
            replay(b, h, n, b_next, h_next, n_next);
            if (failed) break;
            if (staged && tid == 0) {
                sTok[0] = next_beta;
                sTok[1] = next_decay;
            }
            __syncthreads();                        // the shared rows are refilled
            b = b_next; h = h_next; n = n_next;
        }
        if (failed || !mixed) break;
        __syncthreads();                            // the list is rebuilt
    }
    if (failed && tid == 0) record_fault(p.status, kFaultUpdateWait, (int)blockIdx.x);
    if (p.late_wait) grid_dep_wait();
}

// Where the column kernel (update_cols.cu) is the faster one; delta-rule kinds.  Of this kernel's gains over it the one
// reduction per eight tokens is small for GDN, whose decay is one multiplication, and the projections do not pay for a replay
// of many tokens; and a head's time is longer, so it loses where all CTAs wait for the last of few.  Time of this kernel over
// that of the other, r = 8 to 32, both I/O types, 148 SMs:
//   at most one tile of 64 columns (V = 80: 80) per SM            1.0 - 1.6   (two tiles per SM: 0.6 - 1.1)
//   GDN, more than 32 tokens, not 128 x 128                       1.0 - 1.2   (8192 heads; 128 x 128 0.75 - 1.0)
//   GDN, 17 to 32 tokens, K = 128, V <= 80                        0.95 - 1.1  (8192 heads; K = 64 0.8 - 1.0, up to 16 tokens 0.75 - 0.95)
//   GDN, one to one and a half rounds of resident CTAs            0.95 - 1.5, median 1.15  (two full rounds 0.86)
//   KDA, the same, V = 64 or K = 64                               0.95 - 1.4, median 1.07  (two full rounds 0.77)
// Ranks above 32 outweigh the replay again, unless there is no room for the stage (bfloat16 rows read from global memory:
// 64 tokens, r = 64, V = 80 1520 us against 1256).  Per-sequence phases: how many sequences flush is not known here, so only
// the first line counts.  A sketch stored in bfloat16 stays with this kernel: the two differ in the last bits of their fp32
// sums, and what a sequence's stored sketch is rounded to (2^-8 beside a boundary) shall not depend on the size of its batch.
static bool update_cols_better(const Ctx* ctx, const Params& p, int n_tot, size_t wave) {
    const size_t heads = (size_t)p.B * p.H;
    if (p.sketch_bf16) return false;
    if (heads * (p.dv == 128 ? 2 : 1) <= (size_t)ctx->sm_count) return true;
    if (p.n_dev != nullptr) return false;
    const bool kda = ctx->cfg.kind == SKETCHSSM_KDA;
    if (heads > wave && 2 * heads <= 3 * wave && (!kda || p.dv == 64 || p.dk == 64)) return true;
    if (kda || (p.R > 32 && (p.stages || ctx->cfg.io_dtype != SKETCHSSM_BF16))) return false;
    return p.dk == 128 && p.dv == 128 ? false : n_tot > (p.dk == 128 ? 16 : 32);
}

template <int KIND, typename IO, int K, int V>
static int launch_update_t(Ctx* ctx, Params p, cudaStream_t stream) {
    const int n_tot = p.n_before + (p.has_token ? 1 : 0);
    const bool mixed = p.n_dev != nullptr;
    if (mixed) p.n_cap = n_tot;        // per-sequence phases: n_before is the largest fill any sequence may have
    if (ctx->sm_count == 0) {
        int sms = 0;
        if ((ctx->last_cuda_error = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->cfg.device)) != cudaSuccess)
            return SKETCHSSM_CUDA_ERROR;
        ctx->sm_count = sms;
    }
    // Staging one head ahead wherever two CTAs per SM fit with the stage, even if more would fit without: flush of 8192 KDA
    // heads with V = 64, L = 16 304 us against 326 (GDN, where three fit, 271 against 317; V = 80 345 against 408).
    UpdateSmem us = make_update_smem<K>(KIND, n_tot, p.R, V, p.L, (int)sizeof(IO), mixed, 1);
    p.stages = us.total + 1024u <= (228u * 1024u) / 2u ? 1 : 0;
    if (!p.stages) us = make_update_smem<K>(KIND, n_tot, p.R, V, p.L, (int)sizeof(IO), mixed, 0);
    if (us.total > 226u * 1024u) return SKETCHSSM_UNSUPPORTED_SHAPE;
    int by_smem = (int)((228u * 1024u) / (us.total + 1024u));
    by_smem = by_smem < 1 ? 1 : by_smem < update_ctas<V>() ? by_smem : update_ctas<V>();
    const size_t wave = (size_t)ctx->sm_count * (size_t)by_smem;
    if (KIND != SKETCHSSM_MAMBA2 && p.update_impl != 4 && (p.update_impl == 5 || update_cols_better(ctx, p, n_tot, wave)))
        return launch_update_cols(ctx, p, stream);
    auto kern = update_kernel<KIND, IO, K, V>;
    if ((ctx->last_cuda_error = unlock_smem(ctx, kern)) != cudaSuccess) return SKETCHSSM_CUDA_ERROR;
    size_t grid = (size_t)p.B * p.H;
    if (grid > wave) grid = wave;
    if ((ctx->last_cuda_error = launch_kernel(kern, dim3((unsigned)grid), dim3(2 * V), us.total, stream, p, p.pdl != 0)) != cudaSuccess)
        return SKETCHSSM_CUDA_ERROR;
    ctx->last_launches = 1;
    return SKETCHSSM_OK;
}

template <int KIND, typename IO>
static int launch_update_shape(Ctx* ctx, const Params& p, cudaStream_t stream) {
    const int K = ctx->cfg.dk, V = ctx->cfg.dv;
    if (K == 128 && V == 128) return launch_update_t<KIND, IO, 128, 128>(ctx, p, stream);
    if (K == 128 && V == 64) return launch_update_t<KIND, IO, 128, 64>(ctx, p, stream);
    if (K == 128 && V == 80) return launch_update_t<KIND, IO, 128, 80>(ctx, p, stream);
    if (K == 64 && V == 64) return launch_update_t<KIND, IO, 64, 64>(ctx, p, stream);
    if (K == 64 && V == 128) return launch_update_t<KIND, IO, 64, 128>(ctx, p, stream);
    return SKETCHSSM_UNSUPPORTED_SHAPE;
}

template <int KIND>
static int launch_update_io(Ctx* ctx, const Params& p, cudaStream_t stream) {
    if (ctx->cfg.io_dtype == SKETCHSSM_BF16) return launch_update_shape<KIND, __nv_bfloat16>(ctx, p, stream);
    return launch_update_shape<KIND, float>(ctx, p, stream);
}

int launch_update(Ctx* ctx, const Params& p, cudaStream_t stream) {
    switch (ctx->cfg.kind) {
        case SKETCHSSM_MAMBA2: return launch_update_io<SKETCHSSM_MAMBA2>(ctx, p, stream);
        case SKETCHSSM_GDN: return launch_update_io<SKETCHSSM_GDN>(ctx, p, stream);
        case SKETCHSSM_KDA: return launch_update_io<SKETCHSSM_KDA>(ctx, p, stream);
    }
    return SKETCHSSM_INVALID_ARG;
}

}  // namespace sketchssm
