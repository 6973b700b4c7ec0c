// hc_noalloc.cu -- hc_spectrum_noalloc: the forward 2D transform of
// hc_spectrum without any device allocation.
//
// Who needs it: code that must not allocate device memory, for instance a
// plugin living inside a host framework that reserves the whole GPU for its
// own pool allocator, or a latency-critical loop where cudaMalloc's implicit
// device synchronisation is not acceptable.  Such callers own their input and
// output buffers but cannot provide the transform's scratch (the row-pass
// intermediate and the twiddle tables).  Here that scratch is one file-scope
// static device array of fixed size, so it exists in every process that loads
// the library, on every GPU the process uses, until the process exits.
//
// The kernels are the library's own row and column FFT passes, launched on
// the static scratch instead of a context workspace.
#include <cuda_runtime.h>

#include <mutex>

#include "hc.h"
#include "hc_kernels.cuh"

namespace {

using hc::cx;
using hc::fx64;
using hc::FxTw;

constexpr int kMaxDevices = 64;
constexpr size_t kInterBytes = (size_t)HC_NOALLOC_MAX_POINTS / 2 * sizeof(cx<double>);
constexpr int kTables = 2 * 4096;  // the table of length N starts at entry N

// Row-transformed intermediate (ny * nx/2 complex doubles at most) followed by
// the twiddle tables of every length (8 .. 4096).
static __device__ __align__(256) unsigned char g_noalloc_scratch[kInterBytes + kTables * sizeof(FxTw)];

std::mutex g_mu;
void* g_addr[kMaxDevices];    // device address of g_noalloc_scratch per device
bool g_tables[kMaxDevices];   // its tables are filled

// Table entry N + m = exp(-2 pi i m / N), m < N: Q62, or FP64 below the
// fixed-point lengths.
__global__ void k_noalloc_tables(FxTw* tab) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < 8 || i >= kTables) return;
  const int N = 1 << (31 - __clz(i)), m = i - N;
  double s, c;
  sincospi(2.0 * (double)m / (double)N, &s, &c);
  if (N >= (1 << hc::kFxMinLog))
    tab[i] = hc::fx_twiddle(__double2ll_rn(c * 0x1p62), __double2ll_rn(s * -0x1p62));
  else
    reinterpret_cast<double2*>(tab)[i] = make_double2(c, -s);
}

int ilog2i(int v) {
  int l = 0;
  while ((1 << l) < v) ++l;
  return l;
}

bool pow2_in(int v, int lo, int hi) { return v >= lo && v <= hi && (v & (v - 1)) == 0; }

// One-time set-up per device: the device address of the static scratch (the
// host-side symbol is only a stand-in), the shared-memory opt-in of the two
// kernels launched here, and the twiddle tables.  The tables are constants: they
// are complete before the first call returns.  While s is being captured they
// become part of the captured work instead, and a later call fills them for good.
int setup_device(int dev, cudaStream_t s, void** addr) {
  std::lock_guard<std::mutex> lock(g_mu);
  if (dev < 0 || dev >= kMaxDevices) return HC_EINVAL;
  if (!g_addr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return HC_ECUDA;
    cudaGetLastError();  // a pending error of earlier work is not this set-up's
    hc::allow_smem(hc::k_row_r2c<fx64>);
    hc::allow_smem(hc::k_col_fwd<fx64, 1>);
    if (cudaGetLastError() != cudaSuccess) return HC_ECUDA;
    g_addr[dev] = p;
  }
  *addr = g_addr[dev];
  if (!g_tables[dev]) {
    cudaGetLastError();
    k_noalloc_tables<<<kTables / 256, 256, 0, s>>>(
        reinterpret_cast<FxTw*>(static_cast<unsigned char*>(*addr) + kInterBytes));
    if (cudaGetLastError() != cudaSuccess) return HC_ECUDA;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cs) != cudaSuccess) return HC_ECUDA;
    if (cs == cudaStreamCaptureStatusNone) {
      if (cudaStreamSynchronize(s) != cudaSuccess) return HC_ECUDA;
      g_tables[dev] = true;
    }
  }
  return HC_OK;
}

}  // namespace

extern "C" int hc_spectrum_noalloc(const double* f, double* out, int nx, int ny, void* stream) {
  if (!f || !out) return HC_EINVAL;
  if (!pow2_in(nx, 8, 4096) || !pow2_in(ny, 8, 4096)) return HC_EINVAL;
  if ((size_t)nx * (size_t)ny > (size_t)HC_NOALLOC_MAX_POINTS) return HC_EINVAL;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return HC_ECUDA;
  void* base = nullptr;
  cudaStream_t s = (cudaStream_t)stream;
  int rc = setup_device(dev, s, &base);
  if (rc) return rc;
  // A non-sticky error left pending on this thread by earlier work (the
  // caller's or another library's) is consumed here, so that the check after
  // the launches reports only this call's own launches.
  cudaGetLastError();
  unsigned char* b = static_cast<unsigned char*>(base);
  cx<fx64>* inter = reinterpret_cast<cx<fx64>*>(b);
  const FxTw* tab = reinterpret_cast<const FxTw*>(b + kInterBytes);

  hc::Geo<fx64> g = {};
  g.nx = nx;
  g.ny = ny;
  g.H = nx / 2;
  g.lnx = ilog2i(nx);
  g.lny = ilog2i(ny);
  g.lH = ilog2i(nx / 2);
  // 256-thread column CTAs and 128-thread row CTAs, narrower (to one warp) until
  // there are enough of them for the chip, as a context's default shapes
  int tc = 256 >> (g.lny - 3);
  tc = tc < 1 ? 1 : (tc > 32 ? 32 : tc);
  if (tc > g.H) tc = g.H;
  while (tc > 1 && g.H / tc < 128 && (tc >> 1) << (g.lny - 3) >= 32) tc >>= 1;
  g.tc = tc;
  g.ltc = ilog2i(tc);
  int rpc = 128 >> (g.lnx - 3);
  rpc = rpc < 1 ? 1 : rpc;
  if (rpc > ny) rpc = ny;
  while (rpc > 1 && ny / rpc < 512 && (rpc >> 1) << (g.lnx - 3) >= 32) rpc >>= 1;
  g.rpc = rpc;
  g.lrpc = ilog2i(rpc);
  g.twx = reinterpret_cast<const cx<fx64>*>(tab + nx);
  g.twy = reinterpret_cast<const cx<fx64>*>(tab + ny);

  // Every call rewrites the part of the intermediate that it reads, so nothing
  // carried over from an earlier call is used.  The column pass may start while
  // the row pass drains (it waits before its first read): with the tables kept
  // and the narrower CTAs a 256^2 call takes 26.7 us where four launches in 8 and
  // 32 CTAs took 39 (67 with FP64 passes).  What is left is the latency of one
  // warp's instructions: each thread carries 8 points through three passes.
  hc::k_row_r2c<fx64><<<ny >> g.lrpc, rpc << (g.lnx - 3), (size_t)rpc * nx * sizeof(cx<double>), s>>>(
      g, hc::fxp(f), nullptr, inter, nullptr);
  cudaLaunchAttribute early = {};
  early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  early.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(g.H >> g.ltc);
  cfg.blockDim = dim3(tc << (g.lny - 3));
  cfg.dynamicSmemBytes = (size_t)(ny + (ny >> 3)) * tc * sizeof(cx<double>);
  cfg.stream = s;
  cfg.attrs = &early;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, hc::k_col_fwd<fx64, 1>, g, (const cx<fx64>*)inter, (const cx<fx64>*)nullptr,
                     reinterpret_cast<cx<fx64>*>(out), (cx<fx64>*)nullptr, 0,
                     (hc::SolveState*)nullptr);
  if (cudaGetLastError() != cudaSuccess) return HC_ECUDA;
  return HC_OK;
}
