// Adjoint synthesis / analysis without any device allocation.
//
// cmbws_sht_analysis keeps its workspace (the adjoint Legendre stage's input and
// the coefficients) in buffers the grid allocates on first use.  Some callers cannot allocate device
// memory at that point: host runtimes that hand the library a fixed memory
// budget and forbid cudaMalloc after start-up, or real-time loops that must
// not block on the allocator (cudaMalloc can synchronise the device).
// cmbws_sht_analysis_noalloc serves them from one file-scope __device__ array
// of kScratchBytes (32 MiB), which every GPU that loads the library holds
// until the process exits.
//
// The host cannot use the array's name as a device address (in host code it
// names a host-side stand-in), so the device address is looked up with
// cudaGetSymbolAddress once per device, with that device current, on the
// first call made on the device.  Make that first call before any stream
// capture begins.  The address belongs to the device's CUDA context at that
// time; after cudaDeviceReset the cached address is stale, so the library must
// not be used across a reset.  All calls share the one array and find the
// previous call's contents in it; the kernels overwrite every byte they read,
// so nothing needs clearing, but calls whose kernels overlap on the GPU (other
// streams, other host threads) race and must be serialised by the caller.
#include <mutex>

#include "common.h"

namespace cmbws {
namespace {

constexpr size_t kScratchBytes = size_t(32) << 20;
constexpr int kMaxDevices = 64;

static __device__ __align__(256) unsigned char g_scratch[kScratchBytes];

std::mutex g_mu;
void* g_addr[kMaxDevices] = {nullptr};

int scratch_address(void** out) {
  int dev = -1;
  CMBWS_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) {
    set_error("cmbws_sht_analysis_noalloc: device index %d out of range", dev);
    return CMBWS_ERR_ARG;
  }
  std::lock_guard<std::mutex> lk(g_mu);
  if (!g_addr[dev]) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_scratch);
    if (e != cudaSuccess || !p) {
      set_error("cmbws_sht_analysis_noalloc: cudaGetSymbolAddress failed: %s",
                cudaGetErrorString(e));
      return CMBWS_ERR_CUDA;
    }
    g_addr[dev] = p;
  }
  *out = g_addr[dev];
  return CMBWS_OK;
}

size_t round256(size_t n) { return (n + 255) & ~size_t(255); }

// Scratch of a call.  limit: the documented one, ring spectra, adjoint scratch (FP64: partial sums of
// blocks of 256 ring pairs for up to 4 maps) and coefficients together; pb, ob: what is used, the adjoint
// input of nc maps and the coefficients.
struct Scratch {
  size_t limit, pb, ob;
  int nc;
  bool fits() const { return limit <= kScratchBytes && pb + ob <= kScratchBytes; }
};
Scratch scratch_for(const Grid& g, int prec, int nmaps) {
  const size_t es = prec_size(prec);
  const int64_t nlm = nlm_of(g.lmax);
  const int cm = eo_maps(prec), nc = nmaps < cm ? nmaps : cm;
  const size_t fb = round256((size_t)nmaps * g.nring * (g.lmax + 1) * 2 * es);
  const size_t sb = prec == CMBWS_FP64
                        ? round256((size_t)((g.npair + 255) / 256) * 2 * (nc < 4 ? nc : 4) * nlm * 8)
                        : round256(legendre_adjoint_part_bytes(g, prec, nmaps));
  const size_t ob = round256((size_t)nmaps * nlm * 16);
  return {fb + sb + ob, round256(legendre_adjoint_part_bytes(g, prec, nc)), ob, nc};
}

}  // namespace

bool noalloc_fp64(const Grid& g) { return ringfft_smem_ok(g, CMBWS_FP64) && scratch_for(g, CMBWS_FP64, 1).fits(); }

}  // namespace cmbws

using namespace cmbws;

extern "C" int cmbws_sht_analysis_noalloc(cmbws_grid gh, cmbws_prec prec, const double* map,
                                          double* alm, int nmaps, int weighted, void* stream) {
  clear_error();
  Grid* g = as_grid(gh);
  if (!g || !alm || !map || nmaps < 1) {
    set_error("cmbws_sht_analysis_noalloc: invalid arguments");
    return CMBWS_ERR_ARG;
  }
  if (prec != CMBWS_FP64 && prec != CMBWS_FP32) {
    set_error("cmbws_sht_analysis_noalloc: precision %d is not supported here (CMBWS_FP64 or "
              "CMBWS_FP32 only: the double-float and tensor-core modes build tables on first use)",
              (int)prec);
    return CMBWS_ERR_ARG;
  }
  int dev = -1;
  CMBWS_CUDA(cudaGetDevice(&dev));
  if (dev != g->device) {
    set_error("cmbws_sht_analysis_noalloc: grid was planned on device %d, current device is %d",
              g->device, dev);
    return CMBWS_ERR_ARG;
  }
  if (!ringfft_smem_ok(*g, prec)) {
    set_error("cmbws_sht_analysis_noalloc: ring length %d too large for this precision", g->max_n);
    return CMBWS_ERR_ARG;
  }
  const int64_t nlm = nlm_of(g->lmax);
  const Scratch S = scratch_for(*g, prec, nmaps);
  if (!S.fits()) {
    set_error("cmbws_sht_analysis_noalloc: needs %zu bytes of scratch for nmaps=%d, lmax=%d, "
              "nring=%d; the static scratch holds %zu bytes (use cmbws_sht_analysis)",
              S.limit, nmaps, g->lmax, g->nring, kScratchBytes);
    return CMBWS_ERR_ARG;
  }
  void* base = nullptr;
  CMBWS_TRY(scratch_address(&base));
  unsigned char* part = static_cast<unsigned char*>(base);
  double* out = reinterpret_cast<double*>(part + S.pb);
  cudaStream_t s = (cudaStream_t)stream;
  for (int k = 0; k < nmaps; k += S.nc) {
    const int nm = nmaps - k < S.nc ? nmaps - k : S.nc;
    CMBWS_TRY(ringfft_analysis(*g, prec, nm, map + k * g->npix, weighted, part, s));
    CMBWS_TRY(legendre_adjoint(*g, prec, nm, part, S.pb, out + 2 * k * nlm, s));
  }
  CMBWS_TRY(unpack_alm(*g, nmaps, out, alm, s));
  return CMBWS_OK;
}
