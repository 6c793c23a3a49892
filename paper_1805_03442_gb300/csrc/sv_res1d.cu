// sv_res1d.cu -- the resident 1D step loop (sv_res1d.cuh): the float kernels
// and the host entry points res1d_shape / res1d_launch.
#include "sv_res1d.cuh"

namespace sv {

void* res1d_pick_f(const KParams& kp) { return res_pick<float, 0>(kp); }

namespace {

void* pick(const KParams& kp, int precision) {
  switch (precision) {
    case PREC_FP64: return res1d_pick_d(kp);
    case PREC_FP32_P64:
    case PREC_FP32_PC: return res1d_pick_pc(kp);
    case PREC_FP32_PS: return res1d_pick_ps(kp);
    default: return res1d_pick_f(kp);
  }
}

}  // namespace

// Words of the most blocks any device's shape can have (0: none fits).
size_t res1d_word_bytes(int precision, int64_t N) {
  const bool dbl = precision == PREC_FP64;
  const int64_t own = dbl ? 28 : 60, few = dbl ? kResFewD : kResFewF;
  const int64_t wtot = (N + own - 1) / own;
  if (wtot > (int64_t)kResBlocks * (dbl ? kResWarpsD : kResWarpsF)) return 0;
  size_t g = (size_t)((wtot + few - 1) / few);
  if (g > kResBlocks) g = kResBlocks;
  const size_t nw = dbl ? 2 : 1;
  return sizeof(uint64_t) * 2 * g * (g * 2 * nw + 2 * 8 * nw);
}

ResShape res1d_shape(const KParams& kp, int precision, int64_t N) {
  ResShape r = {0, 0, 0};
  int dev = 0, sms = 0, coop = 0, per = 0;
  if (N < 2 || cudaGetDevice(&dev) != cudaSuccess) return r;
  cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (!coop || sms < 1) return r;
  const bool dbl = precision == PREC_FP64;
  const int own = dbl ? 28 : 60, maxw = dbl ? kResWarpsD : kResWarpsF;
  const int lone = dbl ? kResLoneD : kResLoneF, few = dbl ? kResFewD : kResFewF;
  const int64_t wtot = (N + own - 1) / own;
  const int cap = sms < kResBlocks ? sms : kResBlocks;
  if (wtot > (int64_t)cap * maxw) return r;
  int64_t w = wtot <= lone ? wtot : (wtot + cap - 1) / cap;
  if (wtot > lone && w < few) w = few;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, pick(kp, precision), (int)w * 32, 0) !=
          cudaSuccess || per < 1)
    return r;
  r.wtot = (int)wtot;
  r.threads = (int)w * 32;
  r.blocks = (int)((wtot + w - 1) / w);
  return r;
}

cudaError_t res1d_launch(int precision, const KParams& kp, void* a, void* b, Ctl* ctl,
                         uint64_t* words, int64_t N, const ResShape& r, int nmax,
                         cudaStream_t st) {
  if (r.blocks < 1 || nmax < 1 || nmax > 65536) return cudaErrorInvalidValue;
  int n32 = (int)N, wtot = r.wtot;
  void* args[] = {(void*)&kp, &a, &b, &ctl, &words, &n32, &wtot, &nmax};
  if (r.blocks == 1)
    return cudaLaunchKernel(pick(kp, precision), dim3(1), dim3(r.threads), args, 0, st);
  return cudaLaunchCooperativeKernel(pick(kp, precision), dim3(r.blocks), dim3(r.threads), args, 0,
                                     st);
}

}  // namespace sv
