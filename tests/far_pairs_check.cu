// Host build of the far-pair route (csrc/farpair.cuh) for test_far_pairs_cpu.py:
// the four operators' 2 x 2 blocks of n element pairs from FP64 geometry.
#include <math.h>

#include "../paper_2203_13283_gb300/csrc/farpair.cuh"

using namespace wcs;

// ce, cg: n x (x, y, nx, ny) centres; pe, pg: n x q x (x, y, nx, ny) points;
// out: n x 6 operators (S~, D, D~, N, D and D~ of (f, e)) x 4 (a * 2 + b) x (re, im)
extern "C" void far_pairs(int q, const double* xi, const double* w, double k, double beta, double h, int n,
                          const double* ce, const double* cg, const double* pe, const double* pg, double* out) {
  FarConsts F;
  far_consts(F, q, xi, w, k, beta, h, 20.0);
  for (int i = 0; i < n; ++i) {
    const double *a = ce + 4 * i, *b = cg + 4 * i;
    const FarElem E = far_elem(a[0], a[1], a[2], a[3]), G = far_elem(b[0], b[1], b[2], b[3]);
    FarPoint P[FAR_Q], R[FAR_Q];
    for (int p = 0; p < q; ++p) {
      const double *u = pe + 4 * (i * q + p), *v = pg + 4 * (i * q + p);
      P[p] = far_point(a[0], a[1], a[2], a[3], u[0], u[1], u[2], u[3], h, xi[p] - 0.5);
      R[p] = far_point(b[0], b[1], b[2], b[3], v[0], v[1], v[2], v[3], h, xi[p] - 0.5);
    }
    FarPair<true> o;
    if (q == 4) far_pair<4, true>(F, q, E, G, P, R, o);
    else far_pair<0, true>(F, q, E, G, P, R, o);
    for (int op = 0; op < 6; ++op)
      for (int j = 0; j < 4; ++j) {
        const ffc v = o.value(op, j);
        double* d = out + ((i * 6 + op) * 4 + j) * 2;
        d[0] = (double)v.x.hi + v.x.lo;
        d[1] = (double)v.y.hi + v.y.lo;
      }
  }
}
