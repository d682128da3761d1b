// FP32 engine: generic slab kernel here; the slab kernels specialised for a
// tube length live in their own translation units (compiled in parallel).
#include "tc_engine.cuh"
#include "k_tc.cuh"

namespace tc {

bool slab_setup_f32_112(int n2, int optin, SlabCfg<float>& cfg);
bool slab_setup_f32_168(int n2, int optin, SlabCfg<float>& cfg);

template <>
bool pick_slab<float>(int n2, int n3, int optin, SlabCfg<float>& cfg) {
  switch (n3) {
    case 112: return slab_setup_f32_112(n2, optin, cfg);
    case 168: return slab_setup_f32_168(n2, optin, cfg);
    default: return false;
  }
}

template <>
bool pick_tc<float>(int precision, bool split, TcKernels<float>& k) {
  using namespace umma;
  if (precision == TC_TF32) {
    if (split) {
      k = {k_qcon_tc<kTF32, true>, k_dcon_tc<kTF32, true>, k_zsyn_tc<kTF32, true>, qcon_tc_smem<kTF32, true>(),
           dcon_tc_smem<kTF32, true>(), zsyn_tc_smem<kTF32, true>()};
    } else {
      k = {k_qcon_tc<kTF32, false>, k_dcon_tc<kTF32, false>, k_zsyn_tc<kTF32, false>, qcon_tc_smem<kTF32, false>(),
           dcon_tc_smem<kTF32, false>(), zsyn_tc_smem<kTF32, false>()};
    }
    return true;
  }
  if (precision == TC_BF16) {
    if (split) {
      k = {k_qcon_tc<kBF16, true>, k_dcon_tc<kBF16, true>, k_zsyn_tc<kBF16, true>, qcon_tc_smem<kBF16, true>(),
           dcon_tc_smem<kBF16, true>(), zsyn_tc_smem<kBF16, true>()};
    } else {
      k = {k_qcon_tc<kBF16, false>, k_dcon_tc<kBF16, false>, k_zsyn_tc<kBF16, false>, qcon_tc_smem<kBF16, false>(),
           dcon_tc_smem<kBF16, false>(), zsyn_tc_smem<kBF16, false>()};
    }
    return true;
  }
  return false;
}

template <>
bool pick_gemm<float>(int rp, int r, int n2, bool strided, TcKernels<float>& k) {
  k.zsyn = k_zsyn_f<float>;
  k.zsm = zsyn_f_smem<float>(r);
  k.qsm = qcon_smem_bytes<float>(n2, r, rp);
  // (tiled Q is the faster one at r <= 8: 20 against 26 us on 925 x 153 x 92)
  if (rp == 8 && !strided) {
    k.qcon = k_qcon_f<8>, k.dcon = k_dcon_f<8>, k.qsm = qcon_f_smem<8>(), k.dsm = dcon_f_smem<8>();
  } else if (rp == 8) {
    k.qcon = k_qcon_l<8>, k.dcon = k_dcon_f<8, true>, k.dsm = dcon_f_smem<8>();
  } else if (rp == 16 && !strided) {
    k.qcon = k_qcon_l<16>, k.dcon = k_dcon_f<16>, k.dsm = dcon_f_smem<16>();
  } else if (rp == 32 && !strided) {
    k.qcon = k_qcon_l<32>, k.dcon = k_dcon_f<32>, k.dsm = dcon_f_smem<32>();
  } else {
    return false;
  }
  return true;
}

EngineBase* make_engine_f32() { return new Engine<float>(); }

}  // namespace tc
