// Device-side table builders shared by the translation units of the library.
#pragma once
#include "fft.cuh"

namespace pwf {
inline namespace PWF_KNS {

// Twiddle entries of one (length, direction): stage k >= 1 of radix R after
// NS points holds exp(D 2 pi i r j / (NS R)) at tw_entry(NS, r, j).
inline __device__ void fill_twiddles(float2* tab, int n, int D, int idx) {
  const Sched s = sched_for(n);
  for (int k = 1; k < s.s; k++) {
    const int R = stage_radix(n, D, k), NS = stage_ns(n, D, k), off = stage_twoff(n, D, k);
    const int cnt = (R - 1) * NS;
    if (idx < cnt) {
      const int r = idx / NS + 1, j = idx % NS;
      const long m = ((long)r * j) % ((long)NS * R);
      double sn, cs;
      sincospi(2.0 * (double)m / (double)(NS * R), &sn, &cs);
      tab[off + tw_entry(NS, r, j)] = make_float2((float)cs, (float)(D * sn));
    }
  }
}

}  // namespace PWF_KNS
}  // namespace pwf
