// lqcd_dslash_noalloc: the FP64 Dirac operator of lqcd_dslash without any
// device allocation.
//
// Some callers cannot allocate device memory while they run: an application
// that hands this library a share of a GPU whose memory is owned by its own
// allocator (so a cudaMalloc outside that allocator fails or fragments the
// pool), or code on a latency-critical path where an allocation's cost or
// possible failure is not acceptable.  For them this entry point keeps its
// scratch -- the even / odd copies of the input (then the output), their fixed-point limbs and the small
// tables the kernels read -- in a file-scope device array of
// LQCD_NOALLOC_SCRATCH_BYTES, and the limbs' exponents (170 KB) in another.  Every GPU that loads the library holds
// them until the process exits.
//
// The kernels are those of lqcd_dslash.  An FP64 kernel that decoded the fixed-point links and clover blocks entry by entry
// took 96 us a call on 4^4 and 131 us on 16 x 12^3 with clover (83 and 105 us with links and blocks in FP64); 33 and 53 us so.
#include <cstdio>
#include <mutex>

#include "internal.h"

namespace {

constexpr int kMaxSites = (LQCD_NOALLOC_SCRATCH_BYTES - 512) / 768;  // per parity
static __device__ __align__(256) unsigned char g_noalloc_scratch[LQCD_NOALLOC_SCRATCH_BYTES];
static __device__ int g_noalloc_exponents[2 * kMaxSites];

constexpr int kMaxDevices = 64;
std::mutex g_mu;
void* g_scratch_addr[kMaxDevices] = {nullptr};
int* g_exponents_addr[kMaxDevices] = {nullptr};

// Device addresses of the scratch arrays on the current device.  In host code
// an array's name is only a host-side stand-in, so the addresses are looked up
// once per device (with that device current) and cached.
int scratch_address(void** out, int** exponents) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    lq_set_error("dslash_noalloc: no usable current CUDA device");
    return LQCD_ECUDA;
  }
  std::lock_guard<std::mutex> lk(g_mu);
  if (!g_scratch_addr[dev]) {
    void *p = nullptr, *q = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e == cudaSuccess) e = cudaGetSymbolAddress(&q, g_noalloc_exponents);
    if (e != cudaSuccess || !p || !q) {
      cudaGetLastError();
      lq_set_error(std::string("dslash_noalloc: cudaGetSymbolAddress failed: ") + cudaGetErrorString(e));
      return LQCD_ECUDA;
    }
    g_scratch_addr[dev] = p;
    g_exponents_addr[dev] = (int*)q;
  }
  *out = g_scratch_addr[dev];
  *exponents = g_exponents_addr[dev];
  return 0;
}

}  // namespace

extern "C" int lqcd_dslash_noalloc(lqcd_lattice* L, int field, const lqcd_slab* dom, int dagger, const double* in,
                                   double* out, void* stream) {
  if (!L || !in || !out) {
    lq_set_error("dslash_noalloc: null argument");
    return LQCD_EBADARG;
  }
  const lqcd_slab d = dom ? *dom : lqcd_slab{0, L->dims[0] - 1};
  if (d.t0 < 0 || d.t1 >= L->dims[0] || d.t0 > d.t1) {
    lq_set_error("dslash_noalloc: slab out of range");
    return LQCD_EBADARG;
  }
  if (field < 0 || field >= (int)L->fields.size()) {
    lq_set_error("dslash_noalloc: field index not loaded");
    return LQCD_ENOFIELD;
  }
  // scratch layout: [descriptor 256 B][output pointer 256 B][in_e][in_o][limbs_e][limbs_o]; out replaces in
  const long long n = (long long)(d.t1 - d.t0 + 1) * L->S3h;  // sites per parity
  const size_t vec_bytes = (size_t)n * 12 * sizeof(double2);
  const size_t need = 512 + 4 * vec_bytes;
  if (need > (size_t)LQCD_NOALLOC_SCRATCH_BYTES) {
    char msg[256];
    snprintf(msg, sizeof msg,
             "dslash_noalloc: slab of %lld sites needs %zu bytes of scratch, more than the %d-byte maximum "
             "(use lqcd_dslash)",
             2 * n, need, (int)LQCD_NOALLOC_SCRATCH_BYTES);
    lq_set_error(msg);
    return LQCD_EBADARG;
  }
  void* base = nullptr;
  int* exponents = nullptr;
  int rc = scratch_address(&base, &exponents);
  if (rc) return rc;
  unsigned char* b8 = (unsigned char*)base;
  double2* v[4];
  for (int k = 0; k < 4; k++) v[k] = (double2*)(b8 + 512) + k * n * 12;

  lq::SysDesc s{};
  s.field = field;
  s.t0 = d.t0;
  s.t1 = d.t1;
  s.wrap = (d.t0 == 0 && d.t1 == L->dims[0] - 1 && L->bc != LQCD_BC_OPEN) ? 1 : 0;
  s.tsign = L->bc == LQCD_BC_ANTIPERIODIC ? -1.f : 1.f;
  s.n = (int)n;
  s.cb0 = (int)(d.t0 * L->S3h);
  s.off = 0;
  Batch b;
  b.nsys = 1;
  b.max_n = n;
  b.total = n;
  b.nby = (int)((n + LQ_BLOCK - 1) / LQ_BLOCK);
  b.tblk_ok = L->S3h % 32 == 0 && (d.t1 - d.t0 + 1) % 4 == 0;
  b.sys = (lq::SysDesc*)b8;
  // the first kernel writes the descriptor and every site of the vectors, so no part of the scratch needs to start at zero
  return lq_dslash_fx(L, b, s, dagger != 0, L->csw != 0.0, (const double2*)in, out, (void**)(b8 + 256), v, exponents,
                      exponents + n, (cudaStream_t)stream);
}
