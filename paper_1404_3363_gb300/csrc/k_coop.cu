// Instantiations of the group-per-ray integrators (k_coop.cuh, k_coop64.cuh).
#include "k_coop64.cuh"

namespace ivv {

void launch_coop32(const DevVolume& V, const DevCamera<float>& cam, const DevTF& tf, const IntegrateArgs& a, bool mixed,
                   bool split, const float4* pin, const float4* pout, const int* pblk, const int* pcnt,
                   const int* active, const int* n_active, int* queue_head, float4* out, DevStats* st, int num_sms,
                   cudaStream_t s) {
#define IVV_COOP(PP, MM, SS)                                                                                          \
  do {                                                                                                                \
    static int per_sm = -1;                                                                                           \
    launch_coop_k(k5_coop<PP, MM, SS>, per_sm, V, cam, tf, a, pin, pout, pblk, pcnt, active, n_active, queue_head, out, \
                  st, num_sms, s);                                                                                    \
  } while (0)
  if (V.P == 2) {
    if (mixed) { if (split) IVV_COOP(2, true, true); else IVV_COOP(2, true, false); }
    else { if (split) IVV_COOP(2, false, true); else IVV_COOP(2, false, false); }
  } else {
    if (mixed) { if (split) IVV_COOP(3, true, true); else IVV_COOP(3, true, false); }
    else { if (split) IVV_COOP(3, false, true); else IVV_COOP(3, false, false); }
  }
#undef IVV_COOP
}

void launch_coop64(const DevVolume& V, const DevCamera<double>& cam, const DevTF& tf, const IntegrateArgs& a,
                   const Dbl4* pin, const Dbl4* pout, const int* pblk, const int* pcnt, const int* active,
                   const int* n_active, int* queue_head, float4* out, DevStats* st, int num_sms, cudaStream_t s) {
  static int per_sm[2] = {-1, -1};
  if (V.P == 2)
    launch_coop_k(k5_coop64<2>, per_sm[0], V, cam, tf, a, pin, pout, pblk, pcnt, active, n_active, queue_head, out, st,
                  num_sms, s);
  else
    launch_coop_k(k5_coop64<3>, per_sm[1], V, cam, tf, a, pin, pout, pblk, pcnt, active, n_active, queue_head, out, st,
                  num_sms, s);
}

}  // namespace ivv
