// State-dependent coefficient map, pivot approximation with up to four pivots: one warp per (batch, head).  What it computes
// stands at the top of coef_map.cu:
//   Q = Gram-Schmidt basis of the first m sketch rows;  RU = U Q^T;  Y = S Q^T;  mu = ||S||_F^2 / K;
//   d_g = max((||U_g||^2 - ||RU_g||^2) / mu, 0), D_g = d_g + lambda;  T_P = I + RU^T D^{-1} RU / mu;
//   yy = T_P^{-1} (Y[k] - E^T Omega[k]) / mu,  C[g][k] = sum_j F[g][j] yy_j + (d_g / D_g) Omega[k][g],  F = D^{-1} RU, E = Diag(d) F.
//
// A warp walks its heads alone (no block barrier) and brings the state and the sketch rows into shared memory by 16-byte
// asynchronous copies, two chunks of 4 KB ahead, across head boundaries.  A lane owns a part of a row of a chunk:
// five packed multiply-adds per pair of columns (four probes, the norm) against probe rows that all lanes read together, one
// shuffle per probe for a whole row; rows are 16 bytes longer in shared memory, so that lanes in different rows read different
// banks.  Everything is fp32.
//
// Bound by memory: the state's second reading beside the flush's dirty lines leaving L2.  A CTA per head with the products as mma.sync tiles
// on tf32 parts issued 7.0 k (V = 128: 10.2 k) warp instructions per head in stages between block barriers; this takes 4.4 k (6.4 k; fp32
// maps 3.9 k).  The map of 16384 heads, bfloat16 storage, rank 16, in CTAs of four warps: 183 -> 141 us (128 x 64), 306 -> 218 us (128 x 128); as it is
// now, fp32, under ncu 190 -> 135 us (128 x 64; DRAM 65 %, issue slots 47 %).  Without the products
// of the stream it takes 5 us less, without Gram-Schmidt's sweeps 12, without the columns 29; with the next chunks asked into L2 as
// well, or probe rows read from shared memory by lanes that own half a row (14 warps instead of 12), the same.
#include "internal.cuh"
#include "lanegroup.cuh"

namespace sketchssm {

namespace {

constexpr int kBuffers = 2;            // chunks on their way
// Lanes that share a row (16 or 20 columns each); a chunk is two rows per lane, 4 KB (V = 80: 5 KB).
template <int V>
__host__ __device__ constexpr int pivot_parts() { return V == 128 ? 8 : 4; }
template <int V>
__host__ __device__ constexpr int pivot_rows() { return 2 * 32 / pivot_parts<V>(); }

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// one warp's shared memory (byte offsets)
struct PivotSmem {
    uint32_t s, u, u_stride, q, y, ru, uu, f, e, dd, t, total;
};
template <int K, int V>
__host__ __device__ inline PivotSmem make_pivot_smem(int R, int su) {
    PivotSmem p;
    const uint32_t R4 = (uint32_t)((R + 3) & ~3);
    uint32_t off = 0;
    p.s = off; off += (uint32_t)(kBuffers * pivot_rows<V>() * (V + 4) * 4);
    p.u_stride = (uint32_t)(V * su + 16);
    p.u = off; off += (uint32_t)R * p.u_stride;
    p.q = off; off += (uint32_t)(4 * V * 4);
    p.y = off; off += (uint32_t)(K * 16);
    p.ru = off; off += R4 * 16u;
    p.f = off; off += R4 * 16u;
    p.e = off; off += R4 * 16u;
    p.uu = off; off += R4 * 4u;
    p.dd = off; off += R4 * 4u;
    p.t = off; off += 64u;
    p.total = (off + 15u) & ~15u;
    return p;
}

}  // namespace

// Warps of an SM (the registers hold no more), each a CTA: few heads spread over the SMs, and large ranks leave room for as many warps
// as shared memory holds.  In CTAs of four 64 heads ran on 16 SMs.  Sketch and map from a prefilled state, K = 128, us: CTA per head
// (coef_map.cu) / CTAs of four / of one, and rows of Omega asked for ahead of their use above 16 ranks:
//   V = 128, rank 16, fp32: 64 heads 22.2 / 22.5 / 21.7, 888 43.6 / 38.3 / 37.5;  rank 24: 64 heads 24.5 / 28.4 / 23.7, 888 46.9 / 45.0 / 40.7
//   V = 64,  rank 16, fp32: 4 heads 14.1 / 15.2 / 13.9, 256 21.0 / 20.9 / 20.2;  rank 24: 4 heads 16.4 / 17.9 / 16.2, 888 33.5 / 34.0 / 30.5
constexpr int kPivotWarps = 12;

template <int K, int V, bool BF>
__global__ void __launch_bounds__(32, kPivotWarps) pivot_map_kernel(const Params p) {
    constexpr int kRows = pivot_rows<V>(), PARTS = pivot_parts<V>(), RS = 32 / PARTS, VP = V / PARTS, NB = kBuffers, NC = K / kRows, SU = BF ? 2 : 4;
    constexpr uint32_t kRowBytes = (V + 4) * 4, kChunkBytes = kRows * kRowBytes;
    static_assert(NC >= NB, "the next head's first chunks are requested from this head's last ones");
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x;
    const int R = p.R, H = p.H;
    const PivotSmem sm = make_pivot_smem<K, V>(R, SU);
    unsigned char* base = smem;
    const uint32_t sbase = smem_u32(base);
    float* sQ = reinterpret_cast<float*>(base + sm.q);
    float* sY = reinterpret_cast<float*>(base + sm.y);
    float* sRU = reinterpret_cast<float*>(base + sm.ru);
    float* sUU = reinterpret_cast<float*>(base + sm.uu);
    float* sF = reinterpret_cast<float*>(base + sm.f);
    float* sE = reinterpret_cast<float*>(base + sm.e);
    float* sDD = reinterpret_cast<float*>(base + sm.dd);
    float* sT = reinterpret_cast<float*>(base + sm.t);

    // Heads in descending order, the warps of the grid side by side: what the flush wrote last is still in L2.  A head's rank:
    // the configured one or the caller's (0: it reads its full state and has no map); with per-sequence phases only the
    // sequences that were just flushed get a new map.
    const int heads = p.B * H, stride = (int)gridDim.x;        // (at most 2^24 heads)
    auto rank_of = [&](int bh) -> int {
        if (p.head_rank == nullptr) return R;
        const int r = p.head_rank[bh % H];
        return r < 0 ? 0 : (r > R ? R : r);
    };
    auto settle = [&](int bh) -> int {       // bh, or the warp's next head with a map; negative: none left
        while (bh >= 0 && (rank_of(bh) == 0 || (p.n_dev != nullptr && p.n_dev[bh / H] >= 0))) bh -= stride;
        return bh;
    };
    const int part = lane / RS, row = lane % RS;
    int fill = 0;                                        // buffer of the next chunk to be requested
    auto request = [&](int bh, int c) {            // chunk c of a head, with its sketch rows before the first one
        if (c == 0) {
            const unsigned char* ug = reinterpret_cast<const unsigned char*>(p.sketch) + (size_t)bh * R * (V * SU);
            constexpr int per = V * SU / 16;
            const int n = rank_of(bh) * per;
            for (int i = lane; i < n; i += 32) cp_async16(sbase + sm.u + (uint32_t)(i / per) * sm.u_stride + (uint32_t)(i % per) * 16u, ug + (size_t)i * 16);
        }
        const unsigned char* sg = reinterpret_cast<const unsigned char*>(p.state + (size_t)bh * (K * V)) + (size_t)c * (kRows * V * 4);
        const uint32_t dst = sbase + sm.s + (uint32_t)fill * kChunkBytes;
        constexpr int per = V / 4;
#pragma unroll
        for (int it = 0; it < kRows * per / 32; ++it) {
            const int i = it * 32 + lane;
            cp_async16(dst + (uint32_t)(i / per) * kRowBytes + (uint32_t)(i % per) * 16u, sg + (size_t)i * 16);
        }
        if (++fill == NB) fill = 0;
    };

    int bh = settle(heads - 1 - (int)blockIdx.x);
    if (bh < 0) return;
#pragma unroll
    for (int c = 0; c < NB; ++c) {
        request(bh, c);
        cp_commit();
    }
    int use = 0;                                         // buffer of the next chunk to be read
    while (bh >= 0) {
        const int next = settle(bh - stride);
        const int G = rank_of(bh), m = min(G, p.pivots), h = bh % H;
        cp_wait<NB - 1>();                               // the sketch rows and the first chunk
        __syncwarp();

        // ---- Gram-Schmidt on the first m sketch rows (two sweeps; a row that lies in the span of its predecessors becomes zero) ----
        {
            constexpr int EV = (V + 31) / 32;            // elements per lane; beyond V (V = 80) zero and never stored
            auto on = [&](int e) { return V % 32 == 0 || lane + 32 * e < V; };
            float q[4][EV];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (j < m) {
                    float u[EV], ref = 0.f;
#pragma unroll
                    for (int e = 0; e < EV; ++e) {
                        u[e] = 0.f;
                        if (on(e)) {
                            if constexpr (BF) u[e] = __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(base + sm.u + j * sm.u_stride)[lane + 32 * e]);
                            else u[e] = reinterpret_cast<const float*>(base + sm.u + j * sm.u_stride)[lane + 32 * e];
                        }
                        ref = fmaf(u[e], u[e], ref);
                    }
                    ref = warp_sum(ref);
#pragma unroll
                    for (int sweep = 0; sweep < 2; ++sweep) {
#pragma unroll
                        for (int i = 0; i < j; ++i) {
                            float d = 0.f;
#pragma unroll
                            for (int e = 0; e < EV; ++e) d = fmaf(q[i][e], u[e], d);
                            d = warp_sum(d);
#pragma unroll
                            for (int e = 0; e < EV; ++e) u[e] = fmaf(-d, q[i][e], u[e]);
                        }
                    }
                    float nn = 0.f;
#pragma unroll
                    for (int e = 0; e < EV; ++e) nn = fmaf(u[e], u[e], nn);
                    nn = warp_sum(nn);
                    const float inv = (ref > 0.f && nn > 1e-12f * ref) ? rsqrtf(nn) : 0.f;
#pragma unroll
                    for (int e = 0; e < EV; ++e) q[j][e] = u[e] * inv;
                } else {
#pragma unroll
                    for (int e = 0; e < EV; ++e) q[j][e] = 0.f;
                }
#pragma unroll
                for (int e = 0; e < EV; ++e)
                    if (on(e)) sQ[j * V + lane + 32 * e] = q[j][e];
            }
        }
        __syncwarp();

        // this lane's columns of the probe rows, in registers for the whole head
        f32x2 q2[4][VP / 2];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int c = 0; c < VP / 4; ++c) {
                const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(sQ + j * V + part * VP + 4 * c);
                q2[j][2 * c] = t.x;
                q2[j][2 * c + 1] = t.y;
            }
        // products of the lane's part of a row (pairs c of it from `cols`) with the four probe rows, and its norm
        auto against_probes = [&](auto cols, float* y, f32x2& nrm) {
            f32x2 acc[4];
#pragma unroll
            for (int c = 0; c < VP / 4; ++c) {
                f32x2 s01, s23;
                cols(c, s01, s23);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    acc[j] = c == 0 ? mul2(s01, q2[j][0]) : fma2(s01, q2[j][2 * c], acc[j]);
                    acc[j] = fma2(s23, q2[j][2 * c + 1], acc[j]);
                }
                nrm = fma2(s01, s01, nrm);
                nrm = fma2(s23, s23, nrm);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float lo, hi;
                unpack2(acc[j], lo, hi);
                y[j] = lo + hi;
            }
        };
        // the products of two rows (row, row + RS), four probes each, summed over the lanes that share them -> dst[row][4]
        auto sum_parts = [&](float (&y)[8], float* dst, int rows) {
            int m = 8;
#pragma unroll
            for (int o = 16; o >= RS; o >>= 1) {
                m /= 2;
                const bool upper = (lane & o) != 0;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (i < m) {
                        const float send = upper ? y[i] : y[i + m], keep = upper ? y[i + m] : y[i];
                        y[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                    }
                }
            }
            // lane bits 16, 8 (, 4): second row, second half of the probes (, odd probe)
            const int r = row + (lane & 16 ? RS : 0);
            if (r < rows) {
                if constexpr (PARTS == 4) *reinterpret_cast<float2*>(dst + 4 * r + (lane & 8 ? 2 : 0)) = make_float2(y[0], y[1]);
                else dst[4 * r + (lane & 8 ? 2 : 0) + (lane & 4 ? 1 : 0)] = y[0];
            }
        };

        // ---- RU[g] = <U_g, Q_j>, ||U_g||^2: a chunk of ranks at a time ----
        for (int g0 = 0; g0 < G; g0 += kRows) {
            float y[8], nn[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int g = min(g0 + u * RS + row, G - 1);
                const unsigned char* ur = base + sm.u + (uint32_t)g * sm.u_stride + part * VP * SU;
                f32x2 n2 = pack2(0.f, 0.f);
                against_probes([&](int c, f32x2& s01, f32x2& s23) {
                    if constexpr (BF) {
                        const uint2 t = *reinterpret_cast<const uint2*>(ur + 8 * c);
                        s01 = pack2(__uint_as_float(t.x << 16), __uint_as_float(t.x & 0xffff0000u));
                        s23 = pack2(__uint_as_float(t.y << 16), __uint_as_float(t.y & 0xffff0000u));
                    } else {
                        const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(ur + 16 * c);
                        s01 = t.x;
                        s23 = t.y;
                    }
                }, y + 4 * u, n2);
                float lo, hi;
                unpack2(n2, lo, hi);
                nn[u] = lo + hi;
#pragma unroll
                for (int o = RS; o < 32; o <<= 1) nn[u] += __shfl_xor_sync(0xffffffffu, nn[u], o);
            }
            sum_parts(y, sRU + 4 * g0, G - g0);
            if (part < 2 && g0 + part * RS + row < G) sUU[g0 + part * RS + row] = part ? nn[1] : nn[0];
        }

        // ---- Y = S Q^T and ||S||_F^2, chunk by chunk ----
        f32x2 ss2 = pack2(0.f, 0.f);
        __syncwarp();                                    // the sketch rows have been read: the next head's may come in
#pragma unroll 1
        for (int c = 0; c < NC; ++c) {
            if (c > 0) {
                cp_wait<NB - 1>();
                __syncwarp();
            }
            const unsigned char* sr = base + sm.s + (uint32_t)use * kChunkBytes + (uint32_t)row * kRowBytes + part * VP * 4;
            float y[8];
#pragma unroll
            for (int u = 0; u < 2; ++u)
                against_probes([&](int i, f32x2& s01, f32x2& s23) {
                    const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(sr + u * RS * kRowBytes + 16 * i);
                    s01 = t.x;
                    s23 = t.y;
                }, y + 4 * u, ss2);
            __syncwarp();                                // the buffer has been read
            if (c + NB < NC) request(bh, c + NB);
            else if (next >= 0) request(next, c + NB - NC);
            cp_commit();
            sum_parts(y, sY + 4 * c * kRows, kRows);
            if (++use == NB) use = 0;
        }
        float s_lo, s_hi;
        unpack2(ss2, s_lo, s_hi);
        const float ss = warp_sum(s_lo + s_hi);
        const float mu = ss > 0.f ? ss / (float)K : 1.f, inv_mu = 1.f / mu, lam = p.ridge_lambda;

        // ---- per-rank tables (zero rows up to a multiple of four ranks) ----
        const int G4 = (G + 3) & ~3;
        for (int g = lane; g < G4; g += 32) {
            float4 f = make_float4(0.f, 0.f, 0.f, 0.f), e = f;
            float dd = 0.f;
            if (g < G) {
                const float4 ru = *reinterpret_cast<const float4*>(sRU + 4 * g);
                const float r2 = fmaf(ru.w, ru.w, fmaf(ru.z, ru.z, fmaf(ru.y, ru.y, ru.x * ru.x)));
                const float d = fmaxf((sUU[g] - r2) * inv_mu, 0.f), dinv = 1.f / (d + lam);
                f = make_float4(ru.x * dinv, ru.y * dinv, ru.z * dinv, ru.w * dinv);
                e = make_float4(f.x * d, f.y * d, f.z * d, f.w * d);
                dd = d * dinv;
            }
            *reinterpret_cast<float4*>(sF + 4 * g) = f;
            *reinterpret_cast<float4*>(sE + 4 * g) = e;
            sDD[g] = dd;
        }
        __syncwarp();
        // ---- T_P^{-1} / mu: lane (gq, b) holds column b of [T_P | I] for the ranks g = gq mod 4, the four groups are summed by
        // shuffles; Gauss-Jordan with lane = column (symmetric positive definite, eigenvalues >= 1: no pivoting) ----
        {
            const int b = lane & 7, gq = lane >> 3;
            float t[4] = {0.f, 0.f, 0.f, 0.f};
            for (int g = gq; g < G; g += 4) {
                const float4 ru = *reinterpret_cast<const float4*>(sRU + 4 * g);
                const float w = b < 4 ? sF[4 * g + b] : 0.f;
                t[0] = fmaf(ru.x, w, t[0]);
                t[1] = fmaf(ru.y, w, t[1]);
                t[2] = fmaf(ru.z, w, t[2]);
                t[3] = fmaf(ru.w, w, t[3]);
            }
#pragma unroll
            for (int o = 8; o < 32; o <<= 1)
#pragma unroll
                for (int a = 0; a < 4; ++a) t[a] += __shfl_xor_sync(0xffffffffu, t[a], o);
#pragma unroll
            for (int a = 0; a < 4; ++a) t[a] = b < 4 ? fmaf(t[a], inv_mu, a == b ? 1.f : 0.f) : (a == b - 4 ? 1.f : 0.f);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float f[4];
#pragma unroll
                for (int a = 0; a < 4; ++a) f[a] = __shfl_sync(0xffffffffu, t[a], c, 8);
                t[c] *= 1.f / f[c];
#pragma unroll
                for (int a = 0; a < 4; ++a)
                    if (a != c) t[a] = fmaf(-f[a], t[c], t[a]);
            }
            if (lane >= 4 && lane < 8) {
#pragma unroll
                for (int a = 0; a < 4; ++a) sT[4 * a + lane - 4] = t[a] * inv_mu;
            }
        }
        __syncwarp();

        // ---- columns k = lane, lane + 32, .. of C, two at a time (all four at once, their rows of Omega requested before the
        // tables, measured 3 to 6 % slower) ----
        const float* Om = p.omega + (size_t)h * K * R;
        float* Cg = const_cast<float*>(p.coef) + (size_t)bh * R * K;
        __nv_bfloat16* Cg16 = reinterpret_cast<__nv_bfloat16*>(const_cast<float*>(p.coef)) + (size_t)bh * R * K;
        const bool vec = (R & 3) == 0;
#pragma unroll 1
        for (int k = lane; k < K; k += 64) {
            auto om4 = [&](int u, int g0, float (&o)[4]) {
                const float* omk = Om + (size_t)(k + 32 * u) * R;
                if (vec) {
                    ld4(omk + g0, o);
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i) o[i] = g0 + i < G ? omk[g0 + i] : 0.f;
                }
            };
            float y[2][4], yy[2][4];
#pragma unroll
            for (int u = 0; u < 2; ++u) ld4(sY + 4 * (k + 32 * u), y[u]);
            auto pass1 = [&](int g0, const float (&o)[2][4]) {          // y -= E^T Omega[k][:], four ranks
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float e[4];
                    ld4(sE + 4 * (g0 + i), e);
#pragma unroll
                    for (int u = 0; u < 2; ++u)
#pragma unroll
                        for (int j = 0; j < 4; ++j) y[u][j] = fmaf(-e[j], o[u][i], y[u][j]);
                }
            };
            auto pass2 = [&](int g0, const float (&o)[2][4]) {          // the entries of four ranks
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float f[4];
                    ld4(sF + 4 * (g0 + i), f);
                    const float dd = sDD[g0 + i];
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        float c = dd * o[u][i];
#pragma unroll
                        for (int j = 3; j >= 0; --j) c = fmaf(f[j], yy[u][j], c);
                        if (g0 + i < G) {
                            const size_t at = (size_t)(g0 + i) * K + k + 32 * u;
                            if constexpr (BF) Cg16[at] = __float2bfloat16_rn(c);
                            else Cg[at] = c;
                        }
                    }
                }
            };
            auto solve = [&]() {
                float t[4][4];
#pragma unroll
                for (int a = 0; a < 4; ++a) ld4(sT + 4 * a, t[a]);
#pragma unroll
                for (int u = 0; u < 2; ++u)
#pragma unroll
                    for (int a = 0; a < 4; ++a) {
                        float s = 0.f;
#pragma unroll
                        for (int b = 0; b < 4; ++b) s = fmaf(t[a][b], y[u][b], s);
                        yy[u][a] = s;
                    }
            };
            if (G4 <= 16) {      // up to 16 ranks: the rows of Omega are read once and kept in registers for both passes
                float o[4][2][4];
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (4 * c < G4) {
                        om4(0, 4 * c, o[c][0]);
                        om4(1, 4 * c, o[c][1]);
                    }
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (4 * c < G4) pass1(4 * c, o[c]);
                solve();
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (4 * c < G4) pass2(4 * c, o[c]);
            } else {
                // (more: read twice, four ranks ahead of their use)
                auto walk = [&](auto pass) {
                    float a[2][4], b[2][4];
                    om4(0, 0, a[0]);
                    om4(1, 0, a[1]);
                    for (int g0 = 0; g0 < G4; g0 += 8) {
                        const bool more = g0 + 4 < G4;
                        if (more) {
                            om4(0, g0 + 4, b[0]);
                            om4(1, g0 + 4, b[1]);
                        }
                        pass(g0, a);
                        if (g0 + 8 < G4) {
                            om4(0, g0 + 8, a[0]);
                            om4(1, g0 + 8, a[1]);
                        }
                        if (more) pass(g0 + 4, b);
                    }
                };
                walk(pass1);
                solve();
                walk(pass2);
            }
        }
        __syncwarp();                                    // the tables are written again for the next head
        bh = next;
    }
}

template <int K, int V>
static int launch_pivot_kv(Ctx* ctx, const Params& p, cudaStream_t stream) {
    const PivotSmem sm = make_pivot_smem<K, V>(p.R, p.sketch_bf16 ? 2 : 4);
    if (sm.total > 227u * 1024u) return SKETCHSSM_UNSUPPORTED_SHAPE;
    if (ctx->sm_count == 0) {
        int sms = 0;
        if ((ctx->last_cuda_error = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->cfg.device)) != cudaSuccess)
            return SKETCHSSM_CUDA_ERROR;
        ctx->sm_count = sms;
    }
    int ctas = (int)(228u * 1024u / (sm.total + 1024u));
    if (ctas > kPivotWarps) ctas = kPivotWarps;
    const long long heads = (long long)p.B * p.H;
    // With per-sequence phases a CTA for every head: which sequences flush is known to the device alone, and in a fixed stride some warps
    // have three heads of those while others have none.  Mixed step of 4096 heads, CTA per head (coef_map.cu) / in a stride / so:
    // Mamba-2 128 x 64, a quarter flushing, bfloat16 maps 60 / 67 / 55 us, 128 x 128, rank 32, a sixteenth 83 / 98 / 79; GDN 128 x 128, a quarter 115 / 123 / 106.
    long long grid = (long long)ctx->sm_count * ctas;
    if (grid > heads || p.n_dev != nullptr) grid = heads;
    auto kern = p.sketch_bf16 ? pivot_map_kernel<K, V, true> : pivot_map_kernel<K, V, false>;
    if ((ctx->last_cuda_error = unlock_smem(ctx, kern, true)) != cudaSuccess) return SKETCHSSM_CUDA_ERROR;
    kern<<<dim3((unsigned)grid), dim3(32), sm.total, stream>>>(p);
    if ((ctx->last_cuda_error = cudaGetLastError()) != cudaSuccess) return SKETCHSSM_CUDA_ERROR;
    ctx->last_launches += 1;
    return SKETCHSSM_OK;
}

int launch_pivot_map(Ctx* ctx, const Params& p, cudaStream_t stream) {
    const int K = ctx->cfg.dk, V = ctx->cfg.dv;
    if (p.pivots < 1 || (p.pivots > 4 && p.R > 4)) return SKETCHSSM_UNSUPPORTED_SHAPE;
    // By the rank and the state's shape alone: the two kernels differ in the last bits, and what a stored element is rounded to shall not
    // depend on the size of the batch.  Above 24 ranks the sketch rows and two reads of Omega weigh as much as the state of 64 columns,
    // and a warp has them to itself.  Sketch and map from a prefilled state, fp32, CTA per head -> warp per head, us: rank 32, V = 64, 64
    // heads 22.6 -> 22.7, 888 39.2 -> 35.0;  V = 128, 4 heads 24.1 -> 24.6, 64 25.9 -> 25.8, 888 51.5 -> 45.4, 4736 231 -> 200;  V = 80, 4 heads
    // 21.7 -> 22.9, 256 27.0 -> 27.2, 888 50.4 -> 45.7.
    if (p.R > 32 || (p.R > 24 && V == 64)) return SKETCHSSM_UNSUPPORTED_SHAPE;
    if (K == 128 && V == 128) return launch_pivot_kv<128, 128>(ctx, p, stream);
    if (K == 128 && V == 64) return launch_pivot_kv<128, 64>(ctx, p, stream);
    if (K == 128 && V == 80) return launch_pivot_kv<128, 80>(ctx, p, stream);
    if (K == 64 && V == 64) return launch_pivot_kv<64, 64>(ctx, p, stream);
    if (K == 64 && V == 128) return launch_pivot_kv<64, 128>(ctx, p, stream);
    return SKETCHSSM_UNSUPPORTED_SHAPE;
}

}  // namespace sketchssm
