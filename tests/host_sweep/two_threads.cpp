// The host build of the sweeps with a second entry: sweeps in a tensor-core
// precision, whose products have no host stand-in (qsi_zgemm_tc returns
// cudaErrorNotSupported), beside FP64 ones on another thread.
#include "sweep_host.cpp"

// `count` forward sweeps in QSI_FP64_EMU; returns how many asked for a tensor-core
// product (all of them, whatever other threads run).
extern "C" int host_tc_sweeps(int count) {
  int asked = 0;
  for (int k = 0; k < count; ++k) {
    const int n = 2, b = 2;
    std::vector<std::vector<zc>> store(4, std::vector<zc>(n * b * b));
    for (int i = 0; i < n * b; ++i) store[0][i * b + i % b].x = 1.0;
    SweepArrays F;
    F.n = n;
    F.b = b;
    F.batch = 1;
    F.SA = View{store[0].data(), 0};
    F.Aup = View{store[1].data(), 0};
    F.Alo = View{store[2].data(), 0};
    QsiDevStatus status{};
    QsiExec ex;
    ex.precision = QSI_FP64_EMU;
    ex.status = &status;
    asked += qsi_sweep_forward(ex, F) == cudaErrorNotSupported;
  }
  return asked;
}
