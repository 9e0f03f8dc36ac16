// How the teams of the decode kernel (warps that share a head) are laid out.  Plain host code (no CUDA), so that a test can walk it.
#pragma once

namespace sketchssm {

// A CTA of teams of W holds no more heads than an even spread gives an SM (CTAs of up to `least` warps always may) ...
inline long long heads_per_sm(long long heads, int sms) { return (heads + sms - 1) / sms; }
inline bool team_cta_too_large(int warps, int W, int least, long long heads, int sms) { return warps > least && warps / W > heads_per_sm(heads, sms); }
// ... and of the warps that fit an SM only those count that a head would take.
inline int useful_team_warps(int W, long long heads, int sms) { return heads_per_sm(heads, sms) < 64 ? W * (int)heads_per_sm(heads, sms) : 1 << 20; }

}  // namespace sketchssm
