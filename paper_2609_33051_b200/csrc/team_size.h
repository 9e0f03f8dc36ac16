// How many warps of the decode kernel share a head.  Plain host code (no CUDA), so that a test can hold it against measurements.
//
// One warp per head keeps the most heads in flight and needs no barrier.  A team shortens the time of a head: that counts where the
// heads are few, where their stages leave room for few warps, and for full reads of a state beyond L2, whose rows (registers, through
// L1) are then read by warps of which fewer wait for a sweep.  The CTAs of a team kernel hold no more heads than an even spread gives
// an SM (decode.cu), and its full reads have 80 registers (64 spilled up to 372 bytes in Mamba-2's; with K = V = 64 16 to 72, where the
// eight warps more per SM win: 9472 heads 26.8 against 28.7 us).
// All figures: us a launch with 1 / 2 / 4 warps per head, back to back, 148 SMs; `slots`: heads whose stages fit an SM.
#pragma once

namespace sketchssm {

// A CTA of teams of W holds no more heads than an even spread gives an SM (CTAs of up to `least` warps always may) ...
inline long long heads_per_sm(long long heads, int sms) { return (heads + sms - 1) / sms; }
inline bool team_cta_too_large(int warps, int W, int least, long long heads, int sms) { return warps > least && warps / W > heads_per_sm(heads, sms); }
// ... and of the warps that fit an SM only those count that a head would take.
inline int useful_team_warps(int W, long long heads, int sms) { return heads_per_sm(heads, sms) < 64 ? W * (int)heads_per_sm(heads, sms) : 1 << 20; }
// The kernels name their barriers by the team's number, so each CTA holds all 16 that a CTA can have, of an SM's 64.
constexpr int kTeamCtas = 64 / 16;

// Every head reads its state.  h = heads per SM.  Over 396 points (14 kinds, shapes and types, 64 to 9472 heads, 3 to 62 tokens) the rule
// is at worst 1.02 times one warp per head (GDN 128 x 80 beyond L2 1.12), 0.82 of it in the mean:
//   h <= 2: 4.  128 heads: KDA, 128 x 128, 6 fp32 tokens 6.6 / 5.3 / 4.2, GDN, 14 tokens 7.7 / 6.2 / 5.0, Mamba-2, 128 x 64, 62 tokens 10.0 / 6.0 / 4.5
//   h <= 4 (Mamba-2 6, delta rule 5 up to 16 tokens: a team repeats the sweep, a chain): 2.  592 heads: KDA fp32 7.0 / 5.9 / 7.3, GDN 8.0 / 6.7 / 7.9, Mamba-2
//     128 x 64 6.0 / 4.4 / 4.8; 888 heads: Mamba-2 6.0 / 4.9 / 5.4, KDA fp32 7.7 / 8.2 / 8.1
//   few slots: 4 (delta rule with 128 rows, from as many heads per SM as there are slots; else 2: 64 x 128, 30 fp32 tokens, GDN 4736 heads 57 / 56 / 68, KDA 69 / 68 / 75).  Mamba-2, 62 tokens, 8 slots: 1776 heads 30 / 20 / 16, 9472 130 / 135 / 91; KDA, 20
//     fp32 tokens, 6 slots: 888 heads 16 / 13 / 15, 2368 57 / 66 / 44; 128 x 128, 13 slots: Mamba-2, 30 tokens 2368 heads 49 / 32 / 28, GDN, 30 tokens 1776 32 / 35 / 28,
//     4736 79 / 70 / 74
//   a state beyond L2: 2.  GDN 4736 heads 69 / 51 / 56, KDA fp32 3552 54 / 38 / 40, Mamba-2 128 x 64 9472 55 / 51 / 51
//   within L2: 1.  Mamba-2 128 x 64 2368 heads 11.2 / 11.8 / 11.9, GDN 1184 13.8 / 15.9 / 14.2, KDA fp32 1184 15.3 / 16.0 / 13.5 (bfloat16 15.2 / 17.6 / 15.8); but 4 for
//     Mamba-2, 128 x 128, up to 8 heads per SM, 6 fp32 tokens 1184 17.6 / 14.2 / 11.2, and 2 for the delta rule above 20: KDA 64 x 64 4736 23 / 16 / 21
inline int full_read_team(bool mamba2, int n, long long heads, int sms, int slots, int K, int V, long long stream_bytes) {
    const bool wide = K * V == 128 * 128;
    auto up_to = [&](int h) { return heads <= (long long)h * sms; };
    if (up_to(2) || (up_to(3) && (mamba2 || (n <= 16 && K == 128)))) return 4;
    if (up_to(4) || (mamba2 ? up_to(6) && slots >= 10 : up_to(5) && n <= 16)) return 2;
    if (slots < 10) return mamba2 || (K == 128 && !up_to(slots)) ? 4 : 2;
    if (slots < 16 && wide && (mamba2 || (n > 16 && !up_to(6) && up_to(24)))) return 4;
    if (heads * K * V * 4 > stream_bytes) return 2;
    if (mamba2 && wide && up_to(8) && slots < 32) return 4;
    return !mamba2 && !up_to(20) ? 2 : 1;
}

// A rank table: some heads may read their state (rank 0), the others their sketch; which ones is known to the device alone.  A dense head
// takes twice as long as a whole launch without one, and a team's sketched heads cost more than those of single warps: without a dense head |
// with one of twelve.  The lines lie where the two together gain.
//   to one head per SM: 4.  144 heads: Mamba-2, 128 x 80, 4 tokens 4.4 / 5.3 / 4.2 | 7.7 / 5.6 / 4.2, GDN 64 x 64 3.6 / 3.6 / 3.3 | 4.1 / 3.5 / 3.3, KDA, 30 tokens
//     7.3 / 6.1 / 6.3 | 11.0 / 7.7 / 7.0
//   Mamba-2, 128 x 80 and more: to 6 heads per SM 4, to 12 2 (above 16 tokens to 9 where the single warps' stages hold more).  876 heads, 4 tokens 4.1 / 4.2 / 5.5 | 7.7 / 6.3 / 5.7, 28 tokens 7.6 / 6.5 / 6.8 | 10.5 / 8.4 / 6.9 (a
//     table is given for its dense heads); 1200 heads 4.8 / 5.2 / 7.6 | 7.7 / 7.3 / 8.2, 28 tokens 8.1 / 7.2 / 9.9 | 10.6 / 8.8 / 10.2; 1776 5.8 / 6.3 / 8.4 |
//     8.9 / 7.2 / 8.8, 30 tokens and 9 slots 14.0 / 12.8 / 11.8 | 18.8 / 15.3 / 11.8, 28 and 12 9.4 / 10.7 / 10.9 | 11.4 / 14.0 / 11.0
//   the delta rule: to 3 heads per SM and 16 tokens 4, to 12 (9 above 8 tokens) 2.  GDN, 128 x 128: 444 heads 3.9 / 4.0 / 4.2 | 8.0 / 5.1 / 4.9, 12 tokens 4.8 / 4.6 / 5.3 |
//     8.6 / 6.0 / 6.2; 876 4.2 / 4.4 / 6.0 |
//     8.0 / 6.0 / 6.2, 28 tokens 8.2 / 8.7 / 10.6 | 11.1 / 9.1 / 11.0; 1776, 4 tokens 5.8 / 6.5 / 9.1 | 11.8 / 7.7 / 10.1, 12 tokens 8.0 / 10.3 / 12.3 | 10.3 / 12.3 / 12.8
//   smaller states: 128 x 64 2 to 6 (Mamba-2 4 to 3, 2 to 11, to 9 above 16 tokens): 876 heads of Mamba-2 4.1 / 4.2 / 5.4 | 5.8 / 4.7 / 5.4, 1488, 12 tokens 5.8 / 5.8 / 8.3 |
//     7.2 / 6.3 / 8.6, 1776 4.7 / 6.0 / 8.0 | 6.5 / 6.1 / 8.0; 64 x 64 2 to 4: 444 heads of GDN 3.2 / 3.3 / 3.5 | 3.7 / 3.4 / 3.5, 876 3.4 / 3.6 / 5.3 | 3.9 / 3.8 / 5.3
//   a mixed step between three quarters of a head and one and a half per SM: 1.  The flush of the same call starts on the SMs that the decode leaves; spread over
//     all of them by teams it makes the flush's CTAs share SMs.  128 x 128, one sequence in 16 flushing: 108 heads of GDN 14.2 / 14.2 / 14.2, 144 14.2 / 14.3 / 21.1, 192
//     15.0 / 21.3 / 17.4, Mamba-2 144 11.7 / 11.7 / 16.4, 192 12.3 / 16.4 / 13.2, 288 16.2 / 15.0 / 15.7 (without a flush 144 heads 8.5 / 6.4 / 5.3)
inline int rank_table_team(bool mamba2, bool mixed, int n, long long heads, int sms, int slots, int K, int V) {
    auto up_to = [&](int h) { return heads <= (long long)h * sms; };
    if (mixed && 4 * heads > 3ll * sms && 2 * heads <= 3ll * sms) return 1;
    if (up_to(1)) return 4;
    if (K * V < 128 * 64) return up_to(4) ? 2 : 1;
    if (K * V < 128 * 80) return mamba2 && up_to(3) ? 4 : up_to(!mamba2 ? 6 : n > 16 ? 9 : 11) ? 2 : 1;
    if (mamba2) return up_to(6) ? 4 : up_to(n > 16 && slots >= 10 ? 9 : 12) ? 2 : 1;
    return n <= 16 && up_to(3) ? 4 : up_to(n <= 8 ? 12 : 9) ? 2 : 1;
}

// Mamba-2, one rank for all heads: only where long rings and large ranks leave few slots.  128 x 64, rank 32, 16384 heads: 48 tokens (6 slots) 89 / 84 / 85,
// 56 97 / 92 / 95, 62 (5 slots) 118 / 110 / 102; 32 tokens (10 slots) 61 / 62 / 68.
inline int sketch_team(int slots) { return slots <= 5 ? 4 : slots <= 6 ? 2 : 1; }

}  // namespace sketchssm
