// FP64 engine (folded transform, or the generic one past shared memory).
#include "tc_engine.cuh"

namespace tc {

template <>
bool pick_slab<double>(int, int, int, SlabCfg<double>&) {
  return false;
}

template <>
bool pick_tc<double>(int, bool, TcKernels<double>&) {
  return false;
}

template <>
bool pick_gemm<double>(int, int, int, bool, TcKernels<double>&) {
  return false;
}

EngineBase* make_engine_f64() { return new Engine<double>(); }

}  // namespace tc
