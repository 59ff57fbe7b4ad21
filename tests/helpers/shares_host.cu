// Host driver around the share arithmetic of the on-chip samplers' balanced launches, used only by the CPU tests.
// Reads lines "R n_chains n_sweeps i s" from stdin and prints part s of CTA i, "exists chain first end load save", and the
// limit in polls of the wait for a state after `first` sweeps.
#include <cstdio>

#include "../../paper_1810_02821_gb300/csrc/wf_core.cuh"

int main() {
  int R, S, i, s;
  long long n;
  while (std::scanf("%d %lld %d %d %d", &R, &n, &S, &i, &s) == 5) {
    wf::KPart p;
    const bool exists = wf::kpart_of(i, s, R, n, S, &p);
    std::printf("%d %lld %d %d %d %d %lld\n", int(exists), p.c, p.d0, p.d1, int(p.load), int(p.save),
                wf::kawait_polls(p.d0));
  }
  return 0;
}
