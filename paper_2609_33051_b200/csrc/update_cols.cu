// State-update (flush) kernel of the SketchSSM hot path (sm_100a), CUDA cores, delta-rule kinds: a thread per quarter column.
//
// A CTA owns 64 columns (80 when V = 80) of one head's state and four threads share a column, K/4 rows each, in registers.
// The tokens are replayed one by one,  col <- D_s col;  e = beta_s (v_s[j] - <k_s, col>);  col += e k_s,  so a token costs two
// passes over the registers and a decay of the state where update.cu takes eight tokens per reduction.  It has no chains of
// pair sums, triangular substitution and block barriers per eight tokens, though, and a head of 128 columns is two CTAs: it is
// the faster one where the time of a single head counts or where the replay of many tokens outweighs the projections (the
// rule and both sides' times stand at update_cols_better in update.cu).
// Bound by fp32 issue: 3 n + r + 1 multiply-adds per state element, multiply-add pipe 61 % busy, shared-memory data pipe 64 %
// (8192 GDN heads, V = 80, r = 16, 64 bfloat16 tokens, two CTAs of ten warps per SM: 917 us; update.cu 1048 us, 45 %).  Against
// 64-bit results its states are 0.64 to 0.84, its sketches 0.90 to 0.97 as far off as update.cu's (960 layers, about 1e-7).
#include "internal.cuh"
#include "lanegroup.cuh"

namespace sketchssm {
namespace {

constexpr int kParts = 4;               // threads per column

// shared-memory row of K floats split into kParts parts, each padded by 4 floats so that the four
// parts of a warp read from different banks with 128-bit loads
template <int K>
struct PaddedRow {
    static constexpr int RP = K / kParts;
    static constexpr int stride = K + 4 * kParts;
    __host__ __device__ static constexpr int at(int i) { return i + 4 * (i / RP); }
};

struct ColsSmem {
    uint32_t k_off, g_off, v_off, beta_off, dec_off, q_off, om_off, total;
};

template <int K>
__host__ __device__ inline ColsSmem make_cols_smem(int kind, int n_tot, int R4, int kVT) {
    ColsSmem u;
    const int ntok = n_tot > 0 ? n_tot : 1;
    uint32_t off = 0;
    u.k_off = off; off += (uint32_t)(ntok * PaddedRow<K>::stride * 4);
    u.g_off = off; off += kind == SKETCHSSM_KDA ? (uint32_t)(ntok * PaddedRow<K>::stride * 4) : 0u;
    u.v_off = off; off += (uint32_t)(ntok * kVT * 4);
    u.beta_off = off; off += (uint32_t)(((ntok + 3) & ~3) * 4);
    u.dec_off = off; off += (uint32_t)(((ntok + 3) & ~3) * 4);
    u.q_off = off; off += (uint32_t)(PaddedRow<K>::stride * 4);
    u.om_off = off; off += (uint32_t)(kParts * ((K / kParts) * R4 + 4) * 4);
    u.total = off;
    return u;
}

template <int KIND, typename IO, int K, int kVT>
__global__ void __launch_bounds__(kVT * kParts) update_cols_kernel(const Params p) {
    constexpr int kThreads = kVT * kParts;
    using PR = PaddedRow<K>;
    constexpr int RP = PR::RP;
    extern __shared__ __align__(128) unsigned char smem[];

    const int V = p.dv;
    const int R = p.R, H = p.H;
    const int R4 = (R + 3) & ~3;
    const int vtiles = V / kVT;
    const int bh = blockIdx.x / vtiles;
    const int v0 = (blockIdx.x % vtiles) * kVT;
    const int b = bh / H, h = bh % H;
    // (with per-sequence phases beside the decode kernel of the same step, as update_kernel does: then every CTA waits for
    // that kernel at its end)
    if (!p.late_wait) grid_dep_wait();
    grid_dep_launch_dependents();
    // ring fill: the call's n_before, or with per-sequence phases the sequence's own (a sequence whose phase says
    // "decode step" is left alone by this kernel)
    int n_ring = p.n_before;
    if (p.n_dev != nullptr) {
        const int ph = p.n_dev[b];
        if (ph >= 0) {
            if (p.late_wait) grid_dep_wait();
            return;
        }
        n_ring = -ph - 1;
    }
    const int n_tot = n_ring + (p.has_token ? 1 : 0);

    const ColsSmem us = make_cols_smem<K>(KIND, p.n_dev != nullptr ? p.n_cap : n_tot, R4, kVT);
    float* sK = reinterpret_cast<float*>(smem + us.k_off);
    float* sG = reinterpret_cast<float*>(smem + us.g_off);
    float* sV = reinterpret_cast<float*>(smem + us.v_off);
    float* sBeta = reinterpret_cast<float*>(smem + us.beta_off);
    float* sDec = reinterpret_cast<float*>(smem + us.dec_off);
    float* sQ = reinterpret_cast<float*>(smem + us.q_off);
    float* sOm = reinterpret_cast<float*>(smem + us.om_off);

    const int tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5;
    const int part = lane >> 3;                    // 0..3: which quarter of the rows
    const int j = v0 + warp * 8 + (lane & 7);      // this thread's column
    const int jl = j - v0;

    // ---- state tile -> registers (issued first: the long-latency stream) ----
    float col[RP];
    const float* Sg = p.state + (size_t)bh * K * V + (size_t)(part * RP) * V + j;
#pragma unroll
    for (int ii = 0; ii < RP; ++ii) col[ii] = Sg[(size_t)ii * V];

    // ---- ring + current token -> shared memory (fp32) ----
    const unsigned char* rh = p.ring + (size_t)bh * p.rl.head_bytes;
    const IO* rk = reinterpret_cast<const IO*>(rh);
    const IO* rv = reinterpret_cast<const IO*>(rh + p.rl.v_off);
    const float* rbeta = reinterpret_cast<const float*>(rh + p.rl.beta_off);
    for (int idx = tid; idx < n_tot * K; idx += kThreads) {
        const int s = idx / K, i = idx % K;
        float kv, gv = 1.f;
        if (s < n_ring) {
            kv = static_cast<float>(rk[(size_t)s * K + i]);
            if constexpr (KIND == SKETCHSSM_KDA)
                gv = static_cast<float>(reinterpret_cast<const IO*>(rh + p.rl.decay_off)[(size_t)s * K + i]);
        } else {
            kv = static_cast<float>(reinterpret_cast<const IO*>(p.k)[(size_t)bh * K + i]);
            if constexpr (KIND == SKETCHSSM_KDA)
                gv = static_cast<float>(reinterpret_cast<const IO*>(p.decay)[(size_t)bh * K + i]);
        }
        sK[s * PR::stride + PR::at(i)] = kv;
        if constexpr (KIND == SKETCHSSM_KDA) sG[s * PR::stride + PR::at(i)] = gv;
    }
    for (int idx = tid; idx < n_tot * kVT; idx += kThreads) {
        const int s = idx / kVT, c = idx % kVT;
        sV[idx] = s < n_ring ? static_cast<float>(rv[(size_t)s * V + v0 + c])
                             : static_cast<float>(reinterpret_cast<const IO*>(p.v)[(size_t)bh * V + v0 + c]);
    }
    if (tid < n_tot) {
        const int s = tid;
        sBeta[s] = s < n_ring ? rbeta[s] : p.beta[bh];
        if constexpr (KIND != SKETCHSSM_KDA) {
            sDec[s] = s < n_ring ? reinterpret_cast<const float*>(rh + p.rl.decay_off)[s]
                                 : reinterpret_cast<const float*>(p.decay)[bh];
        }
    }
    if (p.q != nullptr) {
        for (int i = tid; i < K; i += kThreads)
            sQ[PR::at(i)] = static_cast<float>(reinterpret_cast<const IO*>(p.q)[(size_t)bh * K + i]);
    }
    if (p.write_sketch) {
        const float* og = p.omega + (size_t)h * K * R;
        for (int idx = tid; idx < K * R4; idx += kThreads) {
            const int i = idx / R4, g = idx % R4;
            sOm[(i / RP) * (RP * R4 + 4) + (i % RP) * R4 + g] = g < R ? og[(size_t)i * R + g] : 0.f;
        }
    }
    __syncthreads();

    {
        f32x2 c2[RP / 2];
#pragma unroll
        for (int i2 = 0; i2 < RP / 2; ++i2) c2[i2] = pack2(col[2 * i2], col[2 * i2 + 1]);
        for (int s = 0; s < n_tot; ++s) {
            const float4* kp = reinterpret_cast<const float4*>(sK + s * PR::stride + part * (RP + 4));
            f32x2 k2[RP / 2];
#pragma unroll
            for (int i4 = 0; i4 < RP / 4; ++i4) {
                const float4 kq = kp[i4];
                k2[2 * i4] = pack2(kq.x, kq.y);
                k2[2 * i4 + 1] = pack2(kq.z, kq.w);
            }
            f32x2 dot01 = pack2(0.f, 0.f), dot23 = dot01;
            if constexpr (KIND == SKETCHSSM_GDN) {
                const float a = sDec[s];
                const f32x2 a2 = pack2(a, a);
#pragma unroll
                for (int i4 = 0; i4 < RP / 4; ++i4) {
                    c2[2 * i4] = mul2(c2[2 * i4], a2);
                    c2[2 * i4 + 1] = mul2(c2[2 * i4 + 1], a2);
                    dot01 = fma2(k2[2 * i4], c2[2 * i4], dot01);
                    dot23 = fma2(k2[2 * i4 + 1], c2[2 * i4 + 1], dot23);
                }
            } else {
                const float4* gp = reinterpret_cast<const float4*>(sG + s * PR::stride + part * (RP + 4));
#pragma unroll
                for (int i4 = 0; i4 < RP / 4; ++i4) {
                    const float4 gq = gp[i4];
                    c2[2 * i4] = mul2(c2[2 * i4], pack2(gq.x, gq.y));
                    c2[2 * i4 + 1] = mul2(c2[2 * i4 + 1], pack2(gq.z, gq.w));
                    dot01 = fma2(k2[2 * i4], c2[2 * i4], dot01);
                    dot23 = fma2(k2[2 * i4 + 1], c2[2 * i4 + 1], dot23);
                }
            }
            float d0, d1, d2, d3;
            unpack2(dot01, d0, d1);
            unpack2(dot23, d2, d3);
            float dot = (d0 + d2) + (d1 + d3);
            dot += __shfl_xor_sync(0xffffffffu, dot, 8);
            dot += __shfl_xor_sync(0xffffffffu, dot, 16);
            const float e = sBeta[s] * (sV[s * kVT + jl] - dot);
            const f32x2 e2 = pack2(e, e);
#pragma unroll
            for (int i2 = 0; i2 < RP / 2; ++i2) c2[i2] = fma2(k2[i2], e2, c2[i2]);
        }
#pragma unroll
        for (int i2 = 0; i2 < RP / 2; ++i2) unpack2(c2[i2], col[2 * i2], col[2 * i2 + 1]);
    }

    // ---- write the updated tile back ----
    if (p.write_state && n_tot > 0) {
        float* So = p.state + (size_t)bh * K * V + (size_t)(part * RP) * V + j;
#pragma unroll
        for (int ii = 0; ii < RP; ++ii) So[(size_t)ii * V] = col[ii];
    }

    // ---- exact output o[j] = <S_new[:, j], q> ----
    if (p.out != nullptr) {
        const float4* qp = reinterpret_cast<const float4*>(sQ + part * (RP + 4));
        float acc = 0.f, odd = 0.f;                 // (two sums of every other row, here and below: half the rounding steps each)
#pragma unroll
        for (int i4 = 0; i4 < RP / 4; ++i4) {
            const float4 qq = qp[i4];
            acc = fmaf(qq.x, col[4 * i4 + 0], acc);
            odd = fmaf(qq.y, col[4 * i4 + 1], odd);
            acc = fmaf(qq.z, col[4 * i4 + 2], acc);
            odd = fmaf(qq.w, col[4 * i4 + 3], odd);
        }
        acc += odd;
        acc += __shfl_xor_sync(0xffffffffu, acc, 8);
        acc += __shfl_xor_sync(0xffffffffu, acc, 16);
        if (part == 0) {
            if (p.out_bf16) reinterpret_cast<__nv_bfloat16*>(p.out)[(size_t)bh * V + j] = __float2bfloat16_rn(acc);
            else reinterpret_cast<float*>(p.out)[(size_t)bh * V + j] = acc;
        }
    }

    // ---- sketch rows U[g, j] = <S_new[:, j], omega_g>, 4 ranks at a time ----
    if (p.write_sketch) {
        const size_t ug = (size_t)bh * R * V + j;
        for (int g0 = 0; g0 < R4; g0 += 4) {
            float a[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
            const float* op = sOm + (size_t)part * (RP * R4 + 4) + g0;
#pragma unroll
            for (int ii = 0; ii < RP; ++ii) {
                const float4 w = *reinterpret_cast<const float4*>(op + ii * R4);
                a[ii & 1][0] = fmaf(w.x, col[ii], a[ii & 1][0]);
                a[ii & 1][1] = fmaf(w.y, col[ii], a[ii & 1][1]);
                a[ii & 1][2] = fmaf(w.z, col[ii], a[ii & 1][2]);
                a[ii & 1][3] = fmaf(w.w, col[ii], a[ii & 1][3]);
            }
            float a0 = a[0][0] + a[1][0], a1 = a[0][1] + a[1][1], a2 = a[0][2] + a[1][2], a3 = a[0][3] + a[1][3];
            a0 += __shfl_xor_sync(0xffffffffu, a0, 8);  a0 += __shfl_xor_sync(0xffffffffu, a0, 16);
            a1 += __shfl_xor_sync(0xffffffffu, a1, 8);  a1 += __shfl_xor_sync(0xffffffffu, a1, 16);
            a2 += __shfl_xor_sync(0xffffffffu, a2, 8);  a2 += __shfl_xor_sync(0xffffffffu, a2, 16);
            a3 += __shfl_xor_sync(0xffffffffu, a3, 8);  a3 += __shfl_xor_sync(0xffffffffu, a3, 16);
            // part p stores rank g0 + p
            const float mine = part == 0 ? a0 : part == 1 ? a1 : part == 2 ? a2 : a3;
            if (g0 + part < R) store_sketch(p, ug + (size_t)(g0 + part) * V, mine);
        }
    }
    if (p.late_wait) grid_dep_wait();
}

template <int KIND, typename IO, int K, int kVT>
int launch_cols_t(Ctx* ctx, Params p, cudaStream_t stream) {
    const int n_tot = p.n_before + (p.has_token ? 1 : 0);
    if (p.n_dev != nullptr) p.n_cap = n_tot;        // per-sequence phases: n_before is the largest fill any sequence may have
    const ColsSmem us = make_cols_smem<K>(KIND, n_tot, (p.R + 3) & ~3, kVT);
    auto kern = update_cols_kernel<KIND, IO, K, kVT>;
    if ((ctx->last_cuda_error = unlock_smem(ctx, kern)) != cudaSuccess) return SKETCHSSM_CUDA_ERROR;
    const dim3 grid((unsigned)((size_t)p.B * p.H * (ctx->cfg.dv / kVT)));
    if ((ctx->last_cuda_error = launch_kernel(kern, grid, dim3(kVT * kParts), us.total, stream, p, p.pdl != 0)) != cudaSuccess)
        return SKETCHSSM_CUDA_ERROR;
    ctx->last_launches = 1;
    return SKETCHSSM_OK;
}

template <int KIND, typename IO>
int launch_cols_shape(Ctx* ctx, const Params& p, cudaStream_t stream) {
    if (ctx->cfg.dk == 128) return ctx->cfg.dv == 80 ? launch_cols_t<KIND, IO, 128, 80>(ctx, p, stream) : launch_cols_t<KIND, IO, 128, 64>(ctx, p, stream);
    return launch_cols_t<KIND, IO, 64, 64>(ctx, p, stream);
}

}  // namespace

int launch_update_cols(Ctx* ctx, const Params& p, cudaStream_t stream) {
    const bool bf = ctx->cfg.io_dtype == SKETCHSSM_BF16;
    if (ctx->cfg.kind == SKETCHSSM_GDN)
        return bf ? launch_cols_shape<SKETCHSSM_GDN, __nv_bfloat16>(ctx, p, stream) : launch_cols_shape<SKETCHSSM_GDN, float>(ctx, p, stream);
    return bf ? launch_cols_shape<SKETCHSSM_KDA, __nv_bfloat16>(ctx, p, stream) : launch_cols_shape<SKETCHSSM_KDA, float>(ctx, p, stream);
}

}  // namespace sketchssm
