// Test-only exports of the FP32 travel-time kernel's shapes.
#include "mlp32.h"

namespace {
template <int H, bool WIDE>
void shape(long long* out) {
  using C = spider::Mlp32<H, WIDE>;
  out[0] = C::kCtas;
  out[1] = C::kThreads;
  out[2] = (long long)C::kSmem;
  out[3] = C::kTile;
}
template <int H>
int shapes(int wide, long long* out) {
  wide ? shape<H, true>(out) : shape<H, false>(out);
  return 0;
}
}  // namespace

extern "C" int mlp32_shape(int H, int wide, long long* out) {
  switch (H) {
    case 32: return shapes<32>(wide, out);
    case 64: return shapes<64>(wide, out);
    case 128: return shapes<128>(wide, out);
    case 256: return shapes<256>(wide, out);
    default: return -1;
  }
}

extern "C" int mlp32_step_is_narrow(int H, long long P, long long n_b, long long nodes, int sms) {
  return spider::narrow_form(H, spider::step_pairs(P, n_b, nodes), sms);
}
