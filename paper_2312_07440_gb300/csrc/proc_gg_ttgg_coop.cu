// g g -> t tbar g g with one warp per event (coop_kernel.cuh): FP64, FP32, and
// the amplitude pass of the FP16-mixed mode's separate colour sum.  (Not the
// BF16 one's: rounding the amplitude vectors to 8 bits turns the last-bit
// differences between two FP32 evaluations into differences of up to 1.5e-3 in
// W', and the mode keeps the results it had.  Its accuracy does not ask for
// that: against FP64, 65,536 events x 2 points, both forms have an rms error of
// 7.3e-4 in W' and a maximum of 5.6e-3, and the warp-per-event form would take
// 1.08 instead of 2.61 ms.)
#include "../../include/rwgt.h"
#include "coop_kernel.cuh"
#include "gen_qcd_gg_ttgg.cuh"
#include "registry.h"

namespace rw {
namespace {
struct CTab {
  __device__ __forceinline__ static short at(int i) { return gg_ttgg::CI[i]; }
};
template <class R>
constexpr int per_thread = (int)(sizeof(coop::Warp<R>) / 32);
static_assert(sizeof(coop::Warp<float>) % 32 == 0 && sizeof(coop::Warp<double>) % 32 == 0, "whole bytes per thread, 16-byte aligned");
constexpr int SLOTS = 1 << (gg_ttgg::NEXT - 1);

}  // namespace

void register_gg_ttgg_coop(std::vector<KernelEntry>& t) {
  t.push_back({RW_GG_TTGG, RW_FP64, 5, (const void*)&coop::k_coop<double, CM_FMA>, 256, 0, per_thread<double>, nullptr, 24});
  t.push_back({RW_GG_TTGG, RW_FP32, 5, (const void*)&coop::k_coop<float, CM_FMA>, 256, 0, per_thread<float>, nullptr, 24});
  t.push_back({RW_GG_TTGG, RW_MIXED_FP16, 5, (const void*)&coop::k_coop<float, CM_STORE_FP16>, 256, 2, per_thread<float>,
               (const void*)&k_colour_tc<gg_ttgg::K, CM_STORE_FP16, SLOTS, CTab>});
}

}  // namespace rw
