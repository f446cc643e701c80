// The launch shapes of the batched solve over amounts of work: prints 1 for each
// property that holds for all of them.
#include <cstdio>

#include "../paper_1305_2418_gb300/csrc/batch_shape.h"

int main() {
  bool first = true, reached = true, once = true, spread = true, least = true;
  for (int nsm : {1, 132, 152})
    for (int ns : {1, 2, 30, 152, 153, 400, 4096})
      for (int lg = 3; lg <= 9; ++lg)
        for (long long extra : {0LL, 64LL, 1000000LL}) {
          const long long vecs = ((long long)ns << (3 * lg - 3)) + extra;
          const BatchShape r = batch_rule(vecs, ns, nsm);
          const long long g = batch_grid(r, vecs, ns, nsm);
          BatchShape c[10];
          const int n = batch_candidates(vecs, ns, nsm, c);
          // the untuned launch is timed, and first
          first = first && n >= 1 && n <= 10 && c[0].threads == r.threads &&
                  batch_grid(c[0], vecs, ns, nsm) == g;
          // every launch of 128/256/512 x 1/2/4 is one of the candidates'
          for (int t : {128, 256, 512})
            for (int b : {1, 2, 4}) {
              bool found = false;
              for (int i = 0; i < n; ++i)
                found = found || (c[i].threads == t &&
                                  batch_grid(c[i], vecs, ns, nsm) ==
                                      batch_grid(BatchShape{t, b}, vecs, ns, nsm));
              reached = reached && found;
            }
          for (int i = 0; i < n; ++i)
            for (int j = 0; j < i; ++j)
              once = once && !(c[i].threads == c[j].threads &&
                               batch_grid(c[i], vecs, ns, nsm) == batch_grid(c[j], vecs, ns, nsm));
          // a chosen shape of 128 threads spreads a small batch as the untuned one does
          if (r.threads == 128)
            spread = spread && batch_grid(BatchShape{128, r.per_sm}, vecs, ns, nsm) == g;
          // no more blocks per SM than the launch fills
          least = least && (r.per_sm == 1 || (long long)nsm * (r.per_sm - 1) < g);
        }
  // one 8^3 and one 16^3: more than one block, 32 items in each
  const BatchShape f = batch_rule(64, 1, 152), g = batch_rule(512, 1, 152);
  const bool tiny = f.threads == 128 && batch_grid(f, 64, 1, 152) == 4 && g.threads == 128 &&
                    batch_grid(g, 512, 1, 152) == 16;
  const BatchShape a = batch_rule(4096, 1, 152), b = batch_rule(32768, 1, 152),
                   d = batch_rule(24 * 32768, 24, 152), e = batch_rule(1 << 21, 96, 152);
  const bool known = a.threads == 128 && batch_grid(a, 4096, 1, 152) == 128 && b.threads == 256 &&
                     batch_grid(b, 32768, 1, 152) == 128 && d.threads == 256 && d.per_sm == 3 &&
                     e.threads == 512 && e.per_sm == 2;
  std::printf("%d %d %d %d %d %d\n", first, reached, once, spread, least, known && tiny);
  return 0;
}
