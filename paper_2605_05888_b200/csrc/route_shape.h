// Launch shape of the router's chain kernel (host code without CUDA, so that it can be checked by itself).
#pragma once

namespace moehub {

// Token warps per CTA (1 to max_tw) for `tokens` tokens in CTAs of `group` tokens per token warp, `split` CTAs beside each
// other per block of tokens, ew warps along the experts, `chains` chains per thread: what takes least, as waves of CTAs times
// what a wave takes - per h the latency of a chain step or the scheduler's warps times their issue slots, whichever is more
// (cycles as measured, see launch_chains_typed), and about 5000 cycles to start, fill the ring and select.  As long as one
// wave holds the batch that is the fewest warps that do.
// (A count of waves times warps alone takes many waves of a single warp wherever that comes out one smaller.  Measured, us,
// so / as here: 32 experts, H 2048, T 7200 70 / 47, T 12000 359 / 67; 60 experts, T 15000 266 / 138; 160 experts, T 985 87 /
// 38; 224 experts, T 960 112 / 42, with H 7168 323 / 122.)
inline int route_token_warps(int tokens, int H, int group, int split, int ew, int chains, int max_tw, int sms) {
  const double latency = chains == 1 ? 4.5 : chains == 2 ? 6.2 : 12.5, issue = chains == 1 ? 2.5 : chains == 2 ? 3.8 : 12.5;
  int tw = 1;
  double best = 1e300;
  for (int i = 1; i <= max_tw; ++i) {
    const long long waves = ((long long)((tokens + (long long)group * i - 1) / ((long long)group * i)) * split + sms - 1) / sms;
    const double per_h = issue * ew * i / 4 > latency ? issue * ew * i / 4 : latency;
    const double cost = (double)waves * (per_h * H + 5000.0);
    if (cost < best) {
      best = cost;
      tw = i;
    }
    if (waves == 1) break;
  }
  return tw;
}

}  // namespace moehub
