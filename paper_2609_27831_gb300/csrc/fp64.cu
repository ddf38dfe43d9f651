// binary64 mode: C = A B for row-major double matrices through the exact
// Ozaki-II path at p = 53, with a cache of the forward's residue planes for
// the backward products dA = dC B^T and dB = A^T dC.
//
// The paper has no backward; the reading used here keeps every residue of the
// forward.  With b_kj ~ b_hat_kj 2^(f_j - t):
//   dA_ik = sum_j dC_ij b_kj ~ 2^-t sum_j (dC_ij 2^f_j) b_hat_kj,
// so D1 = dC diag(2^f) is integerized per row (its own shared exponents) and
// multiplied with the cached planes of B_hat (transposed, unscaled).  With
// a_ik ~ a_hat_ik 2^(e_i - t):
//   dB_kj = sum_i a_ik dC_ij ~ 2^-t sum_i a_hat_ik (2^e_i dC_ij),
// so D2 = diag(2^e) dC is integerized per column and multiplied with the
// cached planes of A_hat (transposed, unscaled).  The forward picks its
// modulus set for inner length max(M, N, K) so that the same planes serve all
// three products.
#include <algorithm>
#include <list>
#include <map>
#include <mutex>
#include <new>
#include <vector>

#include "oz2_internal.h"

namespace oz2 {

namespace {

constexpr int32_t kSentinel = (int32_t)0x80808080;   // exponent of an all-zero line

// double -> one-limb p = 53 format, times 2^shift where shift comes from a
// per-column (axis 1) or per-row (axis 0) exponent array; an element whose
// line exponent is the all-zero sentinel is set to 0 (its partner line is all
// zero, so it contributes nothing).
__global__ void k_f64_to_mp(const double* __restrict__ src, int64_t ld, int rows, int cols,
                            const int32_t* __restrict__ shift, int axis, uint64_t* __restrict__ limbs,
                            int32_t* __restrict__ exps, int8_t* __restrict__ signs) {
  const int64_t n = (int64_t)rows * cols;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int r = (int)(idx / cols), c = (int)(idx - (int64_t)r * cols);
    const double x = src[(int64_t)r * ld + c];
    const uint64_t bits = (uint64_t)__double_as_longlong(x);
    const int be = (int)((bits >> 52) & 0x7ff);
    uint64_t mant = bits & ((1ull << 52) - 1);
    uint64_t sig = 0;
    int e = 0;
    if (be == 0x7ff || (be == 0 && mant == 0)) {
      sig = 0;                                   // zero, Inf, NaN -> 0 (Sec. 10)
    } else if (be == 0) {
      const int lz = __clzll(mant);              // subnormal: normalise
      sig = mant << lz;
      e = -1021 - (lz - 11);
    } else {
      sig = ((1ull << 52) | mant) << 11;
      e = be - 1022;                             // |x| in [2^(e-1), 2^e)
    }
    if (sig && shift) {
      const int32_t s = shift[axis ? c : r];
      if (s == kSentinel) sig = 0;
      else e += s;
    }
    limbs[idx] = sig;
    exps[idx] = sig ? e : 0;
    signs[idx] = (sig && (bits >> 63)) ? 1 : 0;
  }
}

// Plane transpose: src [G][R][src_pitch] (R rows, K valid columns) ->
// dst [G][K][dst_pitch] (K rows, R valid columns); pitches multiples of 8, 16-byte
// aligned.  A block turns 64 x 64 values: a thread reads 8 of two neighbouring rows
// and pairs them, word (k, r / 2) of the tile, and writes 8 neighbouring r of two
// rows k.  Chunks of four words are swizzled by k / 8, so that both the pairs'
// stores and the 16-byte reads meet no bank twice.  Values up to the pitches are
// read and written (zeros past row R); nothing reads them after.  Bound by memory:
// a forward and backward of 4096^2 operands took 11.3 ms with 2-byte accesses of
// 32 x 32 tiles (0.90 ms a transpose) and takes 9.9 so.
__global__ void __launch_bounds__(256) k_transpose_planes(const uint16_t* __restrict__ src, int64_t src_pitch, int R,
                                                          int K, uint16_t* __restrict__ dst, int64_t dst_pitch) {
  __shared__ __align__(16) uint32_t tile[64 * 32];
  const int g = blockIdx.z, r0 = blockIdx.y * 64, k0 = blockIdx.x * 64;
  const uint16_t* s = src + (int64_t)g * R * src_pitch;
  uint16_t* d = dst + (int64_t)g * K * dst_pitch;
  {
    const int kc = threadIdx.x & 7, rp = threadIdx.x >> 3;
    const int r = r0 + 2 * rp, k = k0 + 8 * kc;
    uint4 a = make_uint4(0u, 0u, 0u, 0u), b = a;
    if (k < K && r < R) a = __ldg(reinterpret_cast<const uint4*>(s + (int64_t)r * src_pitch + k));
    if (k < K && r + 1 < R) b = __ldg(reinterpret_cast<const uint4*>(s + (int64_t)(r + 1) * src_pitch + k));
    uint32_t* t = tile + 8 * kc * 32 + (((rp >> 2) ^ kc) << 2) + (rp & 3);
    const uint32_t x[4] = {a.x, a.y, a.z, a.w}, y[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      t[(2 * i) * 32] = __byte_perm(x[i], y[i], 0x5410);
      t[(2 * i + 1) * 32] = __byte_perm(x[i], y[i], 0x7632);
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = threadIdx.x; i < 512; i += 256) {
    const int c = i & 7, kk = i >> 3;
    const int k = k0 + kk, r = r0 + 8 * c;
    if (k < K && r < R)
      *reinterpret_cast<uint4*>(d + (int64_t)k * dst_pitch + r) =
          *reinterpret_cast<const uint4*>(tile + kk * 32 + ((c ^ (kk >> 3)) << 2));
  }
}

cudaError_t to_mp(const double* src, int64_t ld, int rows, int cols, const int32_t* shift, int axis,
                  uint64_t* limbs, int32_t* exps, int8_t* signs, cudaStream_t s) {
  const int64_t n = (int64_t)rows * cols;
  const int blocks = (int)std::min<int64_t>((n + 255) / 256, 148 * 32);
  k_f64_to_mp<<<blocks, 256, 0, s>>>(src, ld, rows, cols, shift, axis, limbs, exps, signs);
  return cudaGetLastError();
}

cudaError_t transpose_planes(const uint16_t* src, int64_t src_pitch, int R, int K, int G, uint16_t* dst,
                             int64_t dst_pitch, cudaStream_t s) {
  dim3 grid((K + 63) / 64, (R + 63) / 64, G);
  k_transpose_planes<<<grid, 256, 0, s>>>(src, src_pitch, R, K, dst, dst_pitch);
  return cudaGetLastError();
}

size_t al(size_t x) { return (x + 255) / 256 * 256; }

// One-limb matrix buffers inside a device allocation.
struct MpBuf {
  uint64_t* limbs = nullptr;
  int32_t* exp = nullptr;
  int8_t* sign = nullptr;
  int rows = 0, cols = 0;
  static size_t bytes(int r, int c) { return al(8ull * r * c) + al(4ull * r * c) + al((size_t)r * c); }
  void place(uint8_t* base, int r, int c) {
    rows = r; cols = c;
    limbs = reinterpret_cast<uint64_t*>(base);
    exp = reinterpret_cast<int32_t*>(base + al(8ull * r * c));
    sign = reinterpret_cast<int8_t*>(base + al(8ull * r * c) + al(4ull * r * c));
  }
  ozaki2_mat mat() const {
    return ozaki2_mat{limbs, exp, sign, cols, (int64_t)rows * cols};
  }
};

}  // namespace

}  // namespace oz2

struct ozaki2_cache_s {
  int64_t M = 0, N = 0, K = 0;
  ozaki2_opts opts{};
  ozaki2_plan fwd = nullptr, bwd_a = nullptr, bwd_b = nullptr;
  oz2::PlanFacts ff{}, fa{}, fb{};
  void* mem = nullptr;          // fwd workspace + A/B conversions
  bool own_mem = false;         // mem is the library's (else its caller's)
  void* mem_bwd = nullptr;      // backward workspaces + dC conversion, the library's
  oz2::MpBuf a, b;
  std::vector<int64_t> key;     // device, shape and options: what a later forward must match to take it over
  cudaEvent_t done = nullptr;   // recorded after every run with this cache
};

namespace oz2 {
namespace {

// Free the memory that a forward and a backward work in, or let go of its caller's.
void cache_drop_memory(ozaki2_cache_s* c) {
  if (c->own_mem || c->mem_bwd) cudaDeviceSynchronize();
  if (c->own_mem) cudaFree(c->mem);
  if (c->mem_bwd) cudaFree(c->mem_bwd);
  c->mem = c->mem_bwd = nullptr;
  c->own_mem = false;
}

int cache_release(ozaki2_cache_s* c) {
  if (!c) return OZ2_EINVAL;
  if (c->mem || c->done) cudaDeviceSynchronize();    // the plans' tables are read by their runs
  cache_drop_memory(c);
  if (c->done) cudaEventDestroy(c->done);
  if (c->fwd) ozaki2_plan_destroy(c->fwd);
  if (c->bwd_a) ozaki2_plan_destroy(c->bwd_a);
  if (c->bwd_b) ozaki2_plan_destroy(c->bwd_b);
  delete c;
  return OZ2_OK;
}

// Retired caches, kept for the next forward of the same shape and options on the
// same device: their plans with the device tables and pinned launch blocks, whose
// making takes several allocations, table uploads and a device-wide wait; never the
// memory that the products work in, which goes back when a cache is retired.
// Bounded per device: at most kPoolCaches caches and kPoolBytes of tables, the
// oldest freed first; all freed by ozaki2_release_cache and when a library
// allocation fails.  A cache that is taken over makes the new stream wait for
// `done`, so its tables and launch blocks are not rewritten before their last
// readers, whatever their stream.
constexpr size_t kPoolCaches = 32;
constexpr size_t kPoolBytes = (size_t)256 << 20;
std::mutex g_pool_mu;
std::list<ozaki2_cache_s*> g_pool;   // oldest first

size_t cache_table_bytes(const ozaki2_cache_s* c) {
  return plan_device_bytes(c->fwd) + plan_device_bytes(c->bwd_a) + plan_device_bytes(c->bwd_b);
}

std::vector<int64_t> cache_key(int64_t M, int64_t N, int64_t K, const ozaki2_opts& o) {
  int dev = -1;
  cudaGetDevice(&dev);
  return {dev, M, N, K, o.guard_bits, o.t_bits, o.engine, o.k_chunk, o.grid, o.schedule, o.timing, o.crt_engine,
          o.res_engine, o.plane_group, o.gemm_tile};
}

// Runs inside a stream capture are neither ordered by nor recorded in `done`
// (an event outside the capture cannot be waited for); their cache is not kept.
bool capturing(cudaStream_t s) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  return cudaStreamIsCapturing(s, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone;
}

// A retired cache of this key, or null; `s` then waits for its last run.
ozaki2_cache_s* pool_take(const std::vector<int64_t>& key, cudaStream_t s) {
  if (capturing(s)) return nullptr;
  ozaki2_cache_s* c = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_pool_mu);
    for (auto it = g_pool.end(); it != g_pool.begin();) {       // the latest one: most likely still in L2
      --it;
      if ((*it)->key == key) {
        c = *it;
        g_pool.erase(it);
        break;
      }
    }
  }
  if (c && cudaStreamWaitEvent(s, c->done, 0) != cudaSuccess) {
    cache_release(c);
    c = nullptr;
  }
  return c;
}

// Keep the plans of a cache that its owner has given back, or free it.
int cache_retire(ozaki2_cache_s* c) {
  if (!c) return OZ2_EINVAL;
  int dev = -1;
  if (!c->done || c->key.empty() || cudaGetDevice(&dev) != cudaSuccess || c->key[0] != dev ||
      cache_table_bytes(c) > kPoolBytes)
    return cache_release(c);
  cache_drop_memory(c);
  std::list<ozaki2_cache_s*> out;
  {
    std::lock_guard<std::mutex> lk(g_pool_mu);
    g_pool.push_back(c);
    size_t n = 0, held = 0;                          // of this device, newest first
    for (auto it = g_pool.end(); it != g_pool.begin();) {
      --it;
      if ((*it)->key[0] != dev) continue;
      ++n;
      held += cache_table_bytes(*it);
      if (n > kPoolCaches || held > kPoolBytes) {
        out.push_back(*it);
        it = g_pool.erase(it);
      }
    }
  }
  for (ozaki2_cache_s* q : out) cache_release(q);
  return OZ2_OK;
}

// Memory from the caller where it gives a function for it, else the library's.
int work_malloc(size_t bytes, ozaki2_alloc_fn alloc, void* user, void** p) {
  if (alloc) *p = alloc(bytes, user);
  else if (dev_malloc(p, bytes) != cudaSuccess) *p = nullptr;
  if (!*p) return OZ2_ENOMEM;
  return (reinterpret_cast<uintptr_t>(*p) & 255u) ? OZ2_EINVAL : OZ2_OK;
}

// A cache with its forward plan: host work only.
int cache_plan(int64_t M, int64_t N, int64_t K, const ozaki2_opts* opts, ozaki2_cache_s** out) {
  if (M <= 0 || N <= 0 || K <= 0) return OZ2_EINVAL;
  if (M > INT32_MAX / 2 || N > INT32_MAX / 2 || K > INT32_MAX / 2) return OZ2_ERANGE;
  auto* c = new (std::nothrow) ozaki2_cache_s();
  if (!c) return OZ2_ENOMEM;
  c->M = M; c->N = N; c->K = K;
  if (opts) c->opts = *opts;
  else ozaki2_opts_default(&c->opts);
  PlanExtra ex;
  ex.inner = std::max(M, std::max(N, K));
  ex.kind = 1;
  int rc = plan_create_ex(M, N, K, 53, &c->opts, ex, &c->fwd);
  if (!rc) rc = plan_query(c->fwd, &c->ff);
  if (rc) { cache_release(c); return rc; }
  *out = c;
  return OZ2_OK;
}

int ensure_fwd_memory(ozaki2_cache_s* c, ozaki2_alloc_fn alloc, void* user) {
  const int M = (int)c->M, N = (int)c->N, K = (int)c->K;
  const size_t ws = al(c->ff.ws_bytes);
  const int rc = work_malloc(ws + MpBuf::bytes(M, K) + MpBuf::bytes(K, N), alloc, user, &c->mem);
  if (rc) return rc;
  c->own_mem = !alloc;
  auto* base = static_cast<uint8_t*>(c->mem);
  c->a.place(base + ws, M, K);
  c->b.place(base + ws + MpBuf::bytes(M, K), K, N);
  return OZ2_OK;
}

int run_fwd(ozaki2_cache_s* c, const double* A, int64_t lda, const double* B, int64_t ldb, double* Cd,
            int64_t ldc, cudaStream_t s) {
  if (!A || !B || !Cd || lda < c->K || ldb < c->N || ldc < c->N) return OZ2_EINVAL;
  if (to_mp(A, lda, (int)c->M, (int)c->K, nullptr, 0, c->a.limbs, c->a.exp, c->a.sign, s) != cudaSuccess ||
      to_mp(B, ldb, (int)c->K, (int)c->N, nullptr, 0, c->b.limbs, c->b.exp, c->b.sign, s) != cudaSuccess)
    return OZ2_ECUDA;
  ozaki2_problem q{};
  q.M = c->M; q.N = c->N; q.K = c->K; q.p = 53;
  q.A = c->a.mat();
  q.B = c->b.mat();
  q.C = ozaki2_mat{reinterpret_cast<uint64_t*>(Cd), nullptr, nullptr, ldc, 0};
  return plan_run(c->fwd, &q, c->mem, c->ff.ws_bytes, s);
}

int ensure_bwd(ozaki2_cache_s* c) {
  if (c->bwd_b) return OZ2_OK;
  PlanExtra ea;
  ea.force_t = c->ff.t; ea.force_L = c->ff.L; ea.kind = 1; ea.skip_b = true;
  int rc = c->bwd_a ? OZ2_OK : plan_create_ex(c->M, c->K, c->N, 53, &c->opts, ea, &c->bwd_a);   // dA = D1 (M x N) * B_hat^T
  if (!rc) rc = plan_query(c->bwd_a, &c->fa);
  PlanExtra eb;
  eb.force_t = c->ff.t; eb.force_L = c->ff.L; eb.kind = 1; eb.skip_a = true;
  if (!rc) rc = plan_create_ex(c->K, c->N, c->M, 53, &c->opts, eb, &c->bwd_b);   // dB = A_hat^T * D2 (M x N)
  if (!rc) rc = plan_query(c->bwd_b, &c->fb);
  return rc;
}

int run_bwd(ozaki2_cache_s* c, const double* dC, int64_t lddc, double* dA, int64_t ldda, double* dB,
            int64_t lddb, ozaki2_alloc_fn alloc, void* user, cudaStream_t s) {
  if (!dC || lddc < c->N) return OZ2_EINVAL;
  if ((dA && ldda < c->K) || (dB && lddb < c->N)) return OZ2_EINVAL;
  int rc = ensure_bwd(c);
  if (rc) return rc;
  auto* fw = static_cast<uint8_t*>(c->mem);
  void* mem = alloc ? nullptr : c->mem_bwd;
  if (!mem) {
    const size_t bytes = al(c->fa.ws_bytes) + al(c->fb.ws_bytes) + MpBuf::bytes((int)c->M, (int)c->N);
    rc = work_malloc(bytes, alloc, user, &mem);
    if (rc) return rc;
    if (!alloc) c->mem_bwd = mem;
  }
  auto* bw = static_cast<uint8_t*>(mem);
  uint8_t* ws_a = bw;
  uint8_t* ws_b = bw + al(c->fa.ws_bytes);
  MpBuf d;
  d.place(bw + al(c->fa.ws_bytes) + al(c->fb.ws_bytes), (int)c->M, (int)c->N);
  const int32_t* e_fwd = reinterpret_cast<const int32_t*>(fw + c->ff.off_e);
  const int32_t* f_fwd = reinterpret_cast<const int32_t*>(fw + c->ff.off_f);
  const auto* pa_fwd = reinterpret_cast<const uint16_t*>(fw + c->ff.off_pa);
  const auto* pb_fwd = reinterpret_cast<const uint16_t*>(fw + c->ff.off_pb);
  const int M = (int)c->M, N = (int)c->N, K = (int)c->K, G = c->ff.G;
  if (dA) {
    // D1 = dC diag(2^f) ; B-side planes = B_hat planes [G][N][Kp] transposed to [G][K][Np]
    if (to_mp(dC, lddc, M, N, f_fwd, 1, d.limbs, d.exp, d.sign, s) != cudaSuccess) return OZ2_ECUDA;
    if (transpose_planes(pb_fwd, c->ff.Kp, N, K, G, reinterpret_cast<uint16_t*>(ws_a + c->fa.off_pb),
                         c->fa.Kp, s) != cudaSuccess)
      return OZ2_ECUDA;
    ozaki2_problem q{};
    q.M = c->M; q.N = c->K; q.K = c->N; q.p = 53;
    q.A = d.mat();
    q.C = ozaki2_mat{reinterpret_cast<uint64_t*>(dA), nullptr, nullptr, ldda, 0};
    rc = plan_run(c->bwd_a, &q, ws_a, c->fa.ws_bytes, s);
    if (rc) return rc;
  }
  if (dB) {
    // D2 = diag(2^e) dC ; A-side planes = A_hat planes [G][M][Kp] transposed to [G][K][Mp]
    if (to_mp(dC, lddc, M, N, e_fwd, 0, d.limbs, d.exp, d.sign, s) != cudaSuccess) return OZ2_ECUDA;
    if (transpose_planes(pa_fwd, c->ff.Kp, M, K, G, reinterpret_cast<uint16_t*>(ws_b + c->fb.off_pa),
                         c->fb.Kp, s) != cudaSuccess)
      return OZ2_ECUDA;
    ozaki2_problem q{};
    q.M = c->K; q.N = c->N; q.K = c->M; q.p = 53;
    q.B = d.mat();
    q.C = ozaki2_mat{reinterpret_cast<uint64_t*>(dB), nullptr, nullptr, lddb, 0};
    rc = plan_run(c->bwd_b, &q, ws_b, c->fb.ws_bytes, s);
    if (rc) return rc;
  }
  return OZ2_OK;
}

std::mutex g_mu;
std::map<std::vector<int64_t>, ozaki2_cache_s*> g_nocache;   // forwards without a cache handle

}  // namespace

void release_retired_caches() {
  std::list<ozaki2_cache_s*> out;
  {
    std::lock_guard<std::mutex> lk(g_pool_mu);
    out.swap(g_pool);
  }
  for (ozaki2_cache_s* c : out) cache_release(c);
}

}  // namespace oz2

using namespace oz2;

extern "C" {

int ozaki2_dgemm_fwd_alloc(int64_t M, int64_t N, int64_t K, const double* A, int64_t lda, const double* B,
                           int64_t ldb, double* Cd, int64_t ldc, const ozaki2_opts* opts, ozaki2_alloc_fn alloc,
                           void* user, ozaki2_cache* cache_out, void* stream) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  try {
    ozaki2_opts o;
    if (opts) o = *opts;
    else ozaki2_opts_default(&o);
    if (cache_out) *cache_out = nullptr;
    if (!A || !B || !Cd || lda < K || ldb < N || ldc < N) {
      // refused on the host; a size or option that no plan takes is named first
      ozaki2_cache_s* c = nullptr;
      const int rc = cache_plan(M, N, K, &o, &c);
      if (rc) return rc;
      cache_release(c);
      return OZ2_EINVAL;
    }
    if (cache_out) {
      auto key = cache_key(M, N, K, o);
      ozaki2_cache_s* c = pool_take(key, s);
      if (!c) {
        const int rc = cache_plan(M, N, K, &o, &c);
        if (rc) return rc;
      }
      int rc = ensure_fwd_memory(c, alloc, user);
      if (!rc) rc = run_fwd(c, A, lda, B, ldb, Cd, ldc, s);
      if (rc) { cache_release(c); return rc; }
      c->key.clear();                                // kept later only if its runs are recorded
      if (!capturing(s)) {
        if (!c->done && cudaEventCreateWithFlags(&c->done, cudaEventDisableTiming) != cudaSuccess) c->done = nullptr;
        if (c->done && cudaEventRecord(c->done, s) == cudaSuccess) c->key = std::move(key);
      }
      *cache_out = c;
      return OZ2_OK;
    }
    int dev = -1;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(g_mu);
    const std::vector<int64_t> key{dev, M, N, K, o.guard_bits, o.t_bits, o.engine, o.k_chunk, o.grid, o.schedule,
                                    o.crt_engine, o.res_engine};
    auto it = g_nocache.find(key);
    if (it == g_nocache.end()) {
      ozaki2_cache_s* c = nullptr;
      int rc = cache_plan(M, N, K, &o, &c);
      if (rc) return rc;
      rc = ensure_fwd_memory(c, nullptr, nullptr);
      if (rc) { cache_release(c); return rc; }
      it = g_nocache.emplace(key, c).first;
    }
    return run_fwd(it->second, A, lda, B, ldb, Cd, ldc, s);
  } catch (const std::bad_alloc&) {
    return OZ2_ENOMEM;
  }
}

int ozaki2_dgemm_fwd(int64_t M, int64_t N, int64_t K, const double* A, int64_t lda, const double* B,
                     int64_t ldb, double* Cd, int64_t ldc, const ozaki2_opts* opts, ozaki2_cache* cache_out,
                     void* stream) {
  return ozaki2_dgemm_fwd_alloc(M, N, K, A, lda, B, ldb, Cd, ldc, opts, nullptr, nullptr, cache_out, stream);
}

int ozaki2_dgemm_bwd_alloc(ozaki2_cache cache, const double* dC, int64_t lddc, double* dA, int64_t ldda, double* dB,
                           int64_t lddb, ozaki2_alloc_fn alloc, void* user, void* stream) {
  if (!cache) return OZ2_EINVAL;
  try {
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // ordered after the cache's earlier runs, and recorded for the later ones
    const bool ordered = !cache->key.empty() && !capturing(s) && cudaStreamWaitEvent(s, cache->done, 0) == cudaSuccess;
    const int rc = run_bwd(cache, dC, lddc, dA, ldda, dB, lddb, alloc, user, s);
    if (!ordered || cudaEventRecord(cache->done, s) != cudaSuccess) cache->key.clear();
    return rc;
  } catch (const std::bad_alloc&) {
    return OZ2_ENOMEM;
  }
}

int ozaki2_dgemm_bwd(ozaki2_cache cache, const double* dC, int64_t lddc, double* dA, int64_t ldda, double* dB,
                     int64_t lddb, void* stream) {
  return ozaki2_dgemm_bwd_alloc(cache, dC, lddc, dA, ldda, dB, lddb, nullptr, nullptr, stream);
}

int ozaki2_cache_destroy(ozaki2_cache cache) { return cache_retire(cache); }

int ozaki2_retired_caches(int* count, size_t* bytes) {
  if (!count || !bytes) return OZ2_EINVAL;
  std::lock_guard<std::mutex> lk(g_pool_mu);
  *count = (int)g_pool.size();
  *bytes = 0;
  for (const ozaki2_cache_s* c : g_pool) *bytes += cache_table_bytes(c);
  return OZ2_OK;
}

}  // extern "C"
