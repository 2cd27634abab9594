// hpsi2.cu -- batched H psi on two-step transforms: prepares the items of a batch and launches the
// three phases (z inverse, plane pass, z forward).
#include "hpsi2.cuh"

namespace fde {

// Run up to kBatchMax items per launch, as many as fit together; items[i].zstart / pstart are filled here.
template <typename T>
bool launch_hpsi_batch(const HpsiItemDesc<T>* items, int nitems, const GridDims& g, const FftPlans<T>& fp,
                       cudaStream_t st, cudaError_t* status) {
  *status = cudaSuccess;
  for (int i = 0; i < nitems; ++i)
    if (!two_step_grid<T>(g, items[i].sp)) return false;
  const T inv_nr = (T)(1.0 / ((double)g.n1 * g.n2 * g.n3));
  for (int i0 = 0, n = 0; i0 < nitems; i0 += n) {
    n = plane_group<T>(g, items + i0, nitems - i0, kBatchMax);  // at least one: each fits alone
    HpsiBatch<T> B;
    B.n = n;
    int zb = 0, pb = 0;
    for (int j = 0; j < B.n; ++j) {
      const HpsiItemDesc<T>& d = items[i0 + j];
      B.it[j] = HpsiItem<T>{d.sp, d.psi, d.hpsi, d.kin, d.vplane, d.scratch, d.ld, d.nb, zb, pb};
      zb += ceil_div(d.sp.ncol, z_cols<T>()) * d.nb;
      pb += g.n3 * d.nb;
    }
    if (zb == 0) continue;
    {
      ProfScope p("k_zinv", st, 1);
      launch_zinv_cols<T>(g.n3, (unsigned)zb, B, fp.p3.tw, st);
    }
    {
      ProfScope p("k_plane", st, 1);
      *status = launch_plane_pass<T>(g, (unsigned)pb, B, fp, st);
      if (*status != cudaSuccess) return true;
    }
    {
      ProfScope p("k_zfwd", st, 1);
      launch_zfwd_cols<T>(g.n3, (unsigned)zb, B, inv_nr, fp.p3.tw, st);
    }
  }
  return true;
}
template bool launch_hpsi_batch<float>(const HpsiItemDesc<float>*, int, const GridDims&, const FftPlans<float>&,
                                       cudaStream_t, cudaError_t*);
template bool launch_hpsi_batch<double>(const HpsiItemDesc<double>*, int, const GridDims&, const FftPlans<double>&,
                                        cudaStream_t, cudaError_t*);

int plane_density_groups(int nb, int n3) {
  const int g = ceil_div(4 * 152, n3);
  return std::max(1, std::min(g, nb));
}

// The plane pass has one compiled form per grid shape.  The variant calls stay: a pin is taken and
// checked, and no shape reports a tuned variant.
int query_plane_variant(int, int) { return -1; }
bool pin_plane_variant(int v) { return v >= -1 && v < 8; }

}  // namespace fde
