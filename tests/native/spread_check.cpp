// Tile of a small straight-line call (amp_kernel.cu, gen_spread) for programs of
// two devices: each spreads its events over the SMs of its own.  Exit status 1 on a fault.
#include <cstdio>

#include "kernels.h"

int main() {
  int bad = 0;
  for (int sms : {152, 76, 152}) {
    mea::DevProgram p;
    p.num_sms = sms;
    p.n_ext = 5;
    p.n_masks = 12;
    mea::AmpConfig plan;
    plan.H = 12;
    plan.E_cta = 21;
    plan.threads = 256;
    for (long long n : {1LL, 75LL, 76LL, 77LL, 152LL, 153LL, 777LL, 3192LL, 3193LL, 100000LL}) {
      const mea::AmpConfig c = mea::gen_spread(p, plan, n, 4);
      const long long E = n > 21LL * sms - sms ? 21 : (n + sms - 1) / sms;  // a share per SM below the plan's tile
      if (c.E_cta != E || c.threads < c.E_cta * c.H || c.threads > plan.threads) {
        ++bad;
        std::printf("%d SMs, %lld events: %d per CTA, not %lld\n", sms, n, c.E_cta, E);
      }
      if (E < 21 && (c.grid > sms || (long long)c.grid * c.E_cta < n)) ++bad;
    }
  }
  return bad ? 1 : 0;
}
