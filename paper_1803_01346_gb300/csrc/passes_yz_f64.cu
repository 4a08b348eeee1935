// passes_yz_f64.cu - the y and z passes of the FP64 path (passes_fx.cuh); a translation unit of its
// own so that the passes compile in parallel.
#include "passes_fx.cuh"

namespace scfft {
namespace fx {

template <int R1, int R2, bool INV, bool PAD> cudaError_t go_y(const Launch<double>& L, const YArgs& a, int planes) {
  constexpr int TC = R1 >= 8 ? 4 : 8;
  constexpr auto k = ypass_kernel<R1, R2, TC, INV, PAD>;
  const size_t smem = sizeof(fxc) * (R1 * R2 + R2 * (R1 * TC + (TC < 8 ? TC : 0)));
  allow_smem<k>();
  const dim3 grid((a.HX + TC - 1) / TC, planes, 3);
  launch_chained(k, dim3(grid), TC * R1, smem, L.st, a);
  return checked_launch("fx ypass_kernel", grid, TC * R1, smem);
}
template <int R1, int R2, int KIND, bool TB = false> cudaError_t go_z(const Launch<double>& L, const ZArgs& a) {
  constexpr int TC = R1 >= 8 ? 4 : 8;
  constexpr int PADZ = TC < 8 ? TC : 0;
  constexpr int CS = cmax(R2 * (R1 * TC + PADZ), R1 * (R2 * TC + PADZ));
  constexpr auto k = zpass_kernel<R1, R2, TC, KIND, TB>;
  const size_t smem = sizeof(fxc) * (R1 * R2 + 3 * CS);
  allow_smem<k>();
  const int nfull = a.HX / TC, rem = a.HX - nfull * TC;
  const dim3 grid(nfull * a.rows + (a.rows * rem + TC - 1) / TC);
  launch_chained(k, dim3(grid), TC * R1, smem, L.st, a);
  return checked_launch("fx zpass_kernel", grid, TC * R1, smem);
}

cudaError_t launch_y(const Launch<double>& L, bool padded, bool inverse, bool check_done) {
  const Geo& g = L.g;
  YArgs a{};
  a.base = padded ? L.w->Pd : L.w->U;
  a.rows = padded ? 2 * g.ny : g.ny;
  a.sx = padded ? g.sxp : g.sxu;
  a.HX = padded ? g.nx + 1 : g.nx / 2 + 1;
  a.nzs = g.nz;
  a.tw = padded ? L.w->fxp[1] : L.w->fxu[1];
  a.ctrl = L.ctrl;
  a.check_done = check_done ? 1 : 0;
  // the padded forward pass and the curl's unpadded inverse pass of an Eq. 5 iteration: only the
  // planes and rows of Omega's box; in the transposed iteration, the other two passes
  const bool box = padded != inverse ? L.use_box : L.use_tbox;
  a.zoff = box ? L.bz0 : 0;
  a.ylo = box ? L.by0 : 0;
  a.yhi = box ? L.by1 : a.rows;
  const int planes = box ? L.bz1 - L.bz0 : g.nz;
#define YCASE_U(LL, R1, R2) \
  case LL: return inverse ? go_y<R1, R2, true, false>(L, a, planes) : go_y<R1, R2, false, false>(L, a, planes);
#define YCASE_P(LL, R1, R2) \
  case LL: return inverse ? go_y<R1, R2, true, true>(L, a, planes) : go_y<R1, R2, false, true>(L, a, planes);
  if (padded) {
    switch (a.rows) { WIDE_PADDED(YCASE_P) }
  } else {
    switch (a.rows) { WIDE_UNPADDED(YCASE_U) }
  }
#undef YCASE_U
#undef YCASE_P
  return cudaErrorInvalidValue;
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
  a.tw = padded ? w.fxp[2] : w.fxu[2];
  a.kt0 = w.kt[0]; a.kt1 = w.kt[1];
  a.st0 = w.st[0]; a.st1 = w.st[1];
  a.t1 = w.zt[0]; a.t2 = w.zt[1];
  a.e1 = w.ze[0]; a.e2 = w.ze[1];
  a.scale = scale;
  a.kap = reinterpret_cast<const long long*>(w.kap);
  a.ek = w.ek;
  a.nx = g.nx; a.ny = g.ny; a.nz = g.nz;
  a.ctrl = L.ctrl;
  a.check_done = check_done ? 1 : 0;
  // Omega's box: the padded pass's input and the curl's output, or, transposed, the other two
  const bool in = padded ? L.use_box : L.use_tbox, out = padded ? L.use_tbox : L.use_box;
  a.ilo = in ? L.bz0 : 0;
  a.ihi = in ? L.bz1 : Lz;
  a.olo = out ? L.bz0 : 0;
  a.ohi = out ? L.bz1 : Lz;
#define ZCASE_U(LL, R1, R2) case LL: return L.use_tbox ? go_z<R1, R2, 0, true>(L, a) : go_z<R1, R2, 0>(L, a);
#define ZCASE_P(LL, R1, R2) case LL: return L.use_tbox ? go_z<R1, R2, 1, true>(L, a) : go_z<R1, R2, 1>(L, a);
  if (padded) {
    switch (Lz) { WIDE_PADDED(ZCASE_P) }
  } else {
    switch (Lz) { WIDE_UNPADDED(ZCASE_U) }
  }
#undef ZCASE_U
#undef ZCASE_P
  return cudaErrorInvalidValue;
}

}  // namespace fx

INST_PASSES_YZ(double)

}  // namespace scfft
