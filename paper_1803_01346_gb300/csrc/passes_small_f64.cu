// passes_small_f64.cu - launchers of the FP64 passes of small grids (passes_small.cuh).
#include "passes_small.cuh"

namespace scfft {
namespace small {

template <int CIN, int COUT> static cudaError_t go_x(const XArgs<double>& a, cudaStream_t st) {
  const int grid = (a.use_box ? a.bz1 - a.bz0 : a.g.nz) * ((a.use_box ? a.by1 - a.by0 : a.g.ny) / 2);
  if (a.g.nx == 16) launch_chained(xpass_kernel<CIN, COUT, 16>, dim3(grid), 96, 0, st, a);
  else if (a.g.nx == 32) launch_chained(xpass_kernel<CIN, COUT, 32>, dim3(grid), 96, 0, st, a);
  else return cudaErrorInvalidValue;
  return checked_launch("small xpass_kernel", dim3(grid), 96, 0);
}

cudaError_t launch_x(const XArgs<double>& a, int cin, int cout, cudaStream_t st) {
  switch (3 * cin + cout) {
    case 1: return go_x<0, 1>(a, st);
    case 2: return go_x<0, 2>(a, st);
    case 3: return go_x<1, 0>(a, st);
    case 4: return go_x<1, 1>(a, st);
    case 5: return go_x<1, 2>(a, st);
    case 6: return go_x<2, 0>(a, st);
    case 7: return go_x<2, 1>(a, st);
  }
  return cudaErrorInvalidValue;
}

template <int L, bool INV, bool PAD> static cudaError_t go_y(const YArgs& a, cudaStream_t st) {
  constexpr int tc = L == 64 ? 4 : 32 / L;
  const int grid = (3 * a.planes * a.HX + tc - 1) / tc;
  if constexpr (L == 64) launch_chained(ypass64_kernel<INV, PAD>, dim3(grid), 32, 0, st, a);
  else launch_chained(ypass_lanes_kernel<L, INV, PAD>, dim3(grid), 32, 0, st, a);
  return checked_launch("small y pass", dim3(grid), 32, 0);
}

cudaError_t launch_y(const Launch<double>& L, bool padded, bool inverse, bool check_done) {
  const Geo& g = L.g;
  YArgs a{};
  a.base = padded ? L.w->Pd : L.w->U;
  a.rows = padded ? 2 * g.ny : g.ny;
  a.sx = padded ? g.sxp : g.sxu;
  a.HX = padded ? g.nx + 1 : g.nx / 2 + 1;
  a.nzs = g.nz;
  a.tw = padded ? L.w->twp[1] : L.w->twu[1];
  a.ctrl = L.ctrl;
  a.check_done = check_done ? 1 : 0;
  // the padded forward pass and the curl's unpadded inverse pass of an Eq. 5 iteration: only the
  // planes and rows of Omega's box; in the transposed iteration, the other two passes
  const bool box = padded != inverse ? L.use_box : L.use_tbox;
  a.zoff = box ? L.bz0 : 0;
  a.ylo = box ? L.by0 : 0;
  a.yhi = box ? L.by1 : a.rows;
  a.planes = box ? L.bz1 - L.bz0 : g.nz;
  if (!padded) {
    if (a.rows == 16) return inverse ? go_y<16, true, false>(a, L.st) : go_y<16, false, false>(a, L.st);
    if (a.rows == 32) return inverse ? go_y<32, true, false>(a, L.st) : go_y<32, false, false>(a, L.st);
  } else {
    if (a.rows == 32) return inverse ? go_y<32, true, true>(a, L.st) : go_y<32, false, true>(a, L.st);
    if (a.rows == 64) return inverse ? go_y<64, true, true>(a, L.st) : go_y<64, false, true>(a, L.st);
  }
  return cudaErrorInvalidValue;
}

template <int L, int KIND> static cudaError_t go_z(const ZArgs& a, cudaStream_t st) {
  constexpr int tc = L == 64 ? 4 : 32 / L;
  const int grid = (a.rows * a.HX + tc - 1) / tc;
  if constexpr (L == 64) launch_chained(zpass64_kernel, dim3(grid), 96, 0, st, a);
  else launch_chained(zpass_lanes_kernel<L, KIND>, dim3(grid), 96, 0, st, a);
  return checked_launch("small z pass", dim3(grid), 96, 0);
}

cudaError_t launch_z(const Launch<double>& L, bool padded, bool check_done, double scale) {
  const Geo& g = L.g;
  const Work<double>& w = *L.w;
  ZArgs a{};
  a.base = padded ? w.Pd : w.U;
  a.rows = padded ? 2 * g.ny : g.ny;
  a.sx = padded ? g.sxp : g.sxu;
  a.HX = padded ? g.nx + 1 : g.nx / 2 + 1;
  a.nzs = g.nz;
  const int Lz = padded ? 2 * g.nz : g.nz;
  a.tw = padded ? w.twp[2] : w.twu[2];
  a.kt0 = w.kt[0]; a.kt1 = w.kt[1]; a.kt2 = w.kt[2];
  a.st0 = w.st[0]; a.st1 = w.st[1]; a.st2 = w.st[2];
  a.scale = scale;
  a.kap = w.kap;
  a.nx = g.nx; a.ny = g.ny; a.nz = g.nz;
  a.ctrl = L.ctrl;
  a.check_done = check_done ? 1 : 0;
  // Omega's box: the padded pass's input and the curl's output, or, transposed, the other two
  const bool in = padded ? L.use_box : L.use_tbox, out = padded ? L.use_tbox : L.use_box;
  a.ilo = in ? L.bz0 : 0;
  a.ihi = in ? L.bz1 : Lz;
  a.olo = out ? L.bz0 : 0;
  a.ohi = out ? L.bz1 : Lz;
  if (!padded) {
    if (Lz == 16) return go_z<16, 0>(a, L.st);
    if (Lz == 32) return go_z<32, 0>(a, L.st);
  } else {
    if (Lz == 32) return go_z<32, 1>(a, L.st);
    if (Lz == 64) return go_z<64, 1>(a, L.st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace small
}  // namespace scfft
