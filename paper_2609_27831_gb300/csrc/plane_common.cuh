// Pieces shared by the plane GEMM kernels (one SM per 128 x 256 tile, and a
// CTA pair per 256 x 256 tile): the exact reductions of the epilogue and the
// deterministic job order that the producer, MMA and epilogue roles walk.
#pragma once

#include <cstdint>

#include "f32x2.cuh"
#include "oz2_internal.h"
#include "tc_ptx.cuh"

namespace oz2 {
namespace plane {

__device__ __forceinline__ uint32_t barrett32(uint32_t x, uint32_t m, uint32_t mu) {
  uint32_t q = __umulhi(x, mu);
  uint32_t r = x - q * m;
  return r >= m ? r - m : r;
}

// The epilogue's reductions, two values per packed fp32 instruction, all on exact
// integers.  Scalar, with the products in 32-bit Barrett form, they took about 12
// instructions per value (plane GEMMs so and now, ms: 4096^3 p = 2048 68.3 and 65.6,
// 1024^3 p = 256 0.141 and 0.138, 64 ragged products 8.68 and 8.49).
struct EpiMod {
  F32x2 rcp, nm, h;   // 1/m, -m, -(m - 1) / (2 m)
  // x mod m, |x| < 2^24: the quotient is within 0.52 of x / m, the result within
  // 0.52 m of zero
  __device__ __forceinline__ F32x2 centered(F32x2 x) const { return f2_fma(f2_nearest(x, rcp), nm, x); }
  // x mod m in [0, m): (x - (m - 1) / 2) / m is 1 / (2 m) or more away from every
  // half-integer and its nearest integer is floor(x / m); exact while the error of
  // x / m, 2^-23 |x| / m, stays below that: |x| < 2^22
  __device__ __forceinline__ F32x2 floored(F32x2 x) const {
    const F32x2 one = f2_pack(1.f, 1.f);
    return f2_fma(f2_nearest(f2_fma(x, rcp, h), one), nm, x);
  }
};

// One accumulation job: plane `plane` of unit `u` over K chunk `chunk`.
struct Job {
  Unit u;
  int slot;
  int plane;
  int chunk;
  bool first;       // first job of the unit: the MMA overwrites the slot
  bool last;        // last job of the unit: the epilogue writes u_l
  uint32_t kmul;    // write-back multiplier (not last)
};

// Deterministic job order shared by the producer, MMA and epilogue roles:
// units s, s+2, s+4, ... of the CTA's list go to TMEM slot s, and the jobs of
// the two slot streams alternate.
struct JobIter {
  const DevTables* T;
  int ubeg, n;
  int uidx[2], job[2], turn;

  __device__ void init(const DevTables* t, int b, int e) {
    T = t; ubeg = b; n = e - b;
    uidx[0] = 0; uidx[1] = 1; job[0] = job[1] = 0; turn = 0;
  }
  __device__ bool next(Job& j) {
    int s = turn;
    if (uidx[s] >= n) {
      s ^= 1;
      if (uidx[s] >= n) return false;
    }
    const Unit u = T->units[ubeg + uidx[s]];
    const ProbDev& P = T->probs[u.prob];
    const bool two = u.ell >= P.L1;
    const int nch = P.nchunks;
    const int njobs = (two ? 3 : 1) * nch;
    const int jj = job[s];
    const int pi = jj / nch;
    j.u = u;
    j.slot = s;
    j.chunk = jj - pi * nch;
    if (two) {
      const int g0 = P.L1 + 3 * (u.ell - P.L1);
      j.plane = g0 + (pi == 0 ? 0 : (pi == 1 ? 2 : 1));   // P0, Ps, P2
    } else {
      j.plane = u.ell;
    }
    j.first = jj == 0;
    j.last = jj == njobs - 1;
    j.kmul = 1u;
    if (!j.last && j.chunk == nch - 1) {
      const ModConst& mc = T->mods[u.ell];
      j.kmul = pi == 0 ? mc.kmul01 : mc.kmul12;
    }
    if (++job[s] == njobs) {
      job[s] = 0;
      uidx[s] += 2;
    }
    turn = s ^ 1;
    return true;
  }
};

// Debugging aid: the exact sum of each plane product before any reduction,
// when K fits in one accumulation chunk.  A job's accumulator holds its
// plane's sum plus the value the unit's previous job wrote back; that job
// leaves the written-back value in this plane's debug slot, so
// dbg_plane_sums subtracts it, and dbg_write_back leaves the current job's
// for the next plane (Karatsuba order P0, Ps, P2 = planes g0, g0 + 2, g0 + 1).
// Both read the 32 columns at taddr from tensor memory themselves (whole warp)
// and are kept out of line, so that the epilogue's registers and code stay as
// they are when no dump is asked for.
static __device__ __noinline__ void dbg_plane_sums(int32_t* dbg, int plane, bool first, int M, int N, int row,
                                                   int col0, uint32_t taddr) {
  uint32_t v[32];
  tc::tmem_ld32(taddr, v);
  if (row >= M) return;
  int32_t* d = dbg + ((int64_t)plane * M + row) * N + col0;
  for (int i = 0; i < 32 && col0 + i < N; ++i) {
    const int32_t acc = __float2int_rn(__uint_as_float(v[i]));
    d[i] = first ? acc : acc - d[i];
  }
}
static __device__ __noinline__ void dbg_write_back(int32_t* dbg, int plane, int ell, int L1, int M, int N,
                                                   int row, int col0, uint32_t taddr) {
  uint32_t v[32];
  tc::tmem_wait_st();
  tc::tmem_ld32(taddr, v);
  if (row >= M || ell < L1) return;
  const int g0 = L1 + 3 * (ell - L1);
  const int next = plane == g0 ? g0 + 2 : g0 + 1;
  int32_t* d = dbg + ((int64_t)next * M + row) * N + col0;
  for (int i = 0; i < 32 && col0 + i < N; ++i) d[i] = __float2int_rn(__uint_as_float(v[i]));
}

// A job's epilogue constants, gathered before its accumulator is ready (the
// loads run while the epilogue waits for the slot; the chunk loop then reads
// no global memory but the optional debug dump).
struct EpiConst {
  float mf, rcp, hf;  // m, 1/m, -(m - 1) / (2 m)
  uint32_t mul;       // write-back: the next plane's Karatsuba factor; last job:
                      // kfin M_l^{-1} mod m_l, so that the stored value is the
                      // CRT's v_l = (c mod m_l) M_l^{-1} mod m_l (Sec. 4.4)
  int M, N, row, col0, L1, ell;
  uint16_t* uell;     // u of this modulus
  int32_t* dbg;
};

// v_l tiles of one epilogue warp through shared memory: two 2 KB buffers of
// 32 rows x 64 bytes in the 64-byte swizzle (16-byte chunk q of row r at
// r 64 + 16 (q ^ ((r >> 1) & 3)): the eight rows of a store phase hit eight
// different bank groups), each written to u by one TMA store.  map is null
// when u's rows are not 16-byte multiples; then the warp writes the staged
// tile row by row (store_tile_rows).
struct UStage {
  const CUtensorMap* map;
  uint32_t sbuf;      // shared address of the warp's two buffers
  uint32_t n;         // tiles staged so far (warp-uniform)
};

__device__ __forceinline__ EpiConst epi_const(const DevTables& T, const Job& j, int row, int col0) {
  const ProbDev& P = T.probs[j.u.prob];
  const ModConst mc = T.mods[j.u.ell];
  EpiConst e;
  e.mf = (float)mc.m;
  e.rcp = mc.rcp;
  e.hf = -0.5f * (e.mf - 1.f) / e.mf;
  e.M = P.M;
  e.N = P.N;
  e.row = row;
  e.col0 = col0;
  e.L1 = P.L1;
  e.ell = j.u.ell;
  e.uell = P.u + (int64_t)j.u.ell * P.upitch;
  e.dbg = P.dbg_prods;
  e.mul = j.last ? barrett32(mc.kfin * __ldg(crt_view(T.crt_pool, P).Minv + j.u.ell), mc.m, mc.mu) : j.kmul;
  return e;
}

// A staged 32 x 32 tile of v_l (the 64-byte swizzle above) to u where its rows
// are only 2-byte aligned (N not a multiple of 8: no TMA store can reach
// them).  Half a warp takes a row, a lane the two values of a staged word, in
// two 2-byte stores.  What bounds it is the sectors a store instruction
// touches: two rows here (4 to 6 sectors of 32 bytes), where a thread storing
// its own row touched 32 (plane GEMMs of 1531 x 1093 x 1777, p = 512: 2.39 ->
// 1.14 ms, 1.11 with N = 1096 and the TMA store; 64 uneven problems 23.3 -> 9.0
// ms).  Pairing values into aligned words across lanes (a shuffle, one 4-byte
// store and the row's two ends on their own) was slower: 1.40 and 11.5 ms.
static __device__ __noinline__ void store_tile_rows(uint16_t* uell, uint32_t buf, int row0, int col, int M, int N) {
  const int lane = threadIdx.x & 31, c = lane & 15;
  const int c0 = col + 2 * c;
  const bool in0 = c0 < N, in1 = c0 + 1 < N;
  uint16_t* dst = uell + (int64_t)(row0 + (lane >> 4)) * N + c0;
#pragma unroll
  for (int s = 0; s < 16; ++s) {
    const int r = 2 * s + (lane >> 4);
    uint32_t w;
    asm volatile("ld.shared.b32 %0, [%1];"
                 : "=r"(w)
                 : "r"(buf + (uint32_t)(r * 64 + 16 * ((c >> 2) ^ (s & 3)) + 4 * (c & 3)))
                 : "memory");
    if (row0 + r < M) {
      if (in0) dst[0] = (uint16_t)w;
      if (in1) dst[1] = (uint16_t)(w >> 16);
    }
    dst += 2 * (int64_t)N;
  }
}

// One 32-column chunk of a job's accumulator (v, read from taddr; columns
// e.col0 + cc ..): reduce mod m, then either write the residue back into
// TMEM times the next plane's factor, or store v_l.
__device__ __forceinline__ void epi_chunk(const Job& j, const EpiConst& e, uint32_t (&v)[32], uint32_t taddr,
                                          int cc, UStage& us) {
  const int col = e.col0 + cc;
  if (e.dbg != nullptr) dbg_plane_sums(e.dbg, j.plane, j.first, e.M, e.N, e.row, col, taddr);
  const EpiMod md{f2_pack(e.rcp, e.rcp), f2_pack(-e.mf, -e.mf), f2_pack(e.hf, e.hf)};
  const bool two = e.ell >= e.L1;
  // a factor below 2^14 in halves of 7 bits (x times a half below 2^22), or whole below 2^8
  const float f0 = (float)(two ? e.mul & 127u : e.mul), f1 = (float)(e.mul >> 7);
  const F32x2 m0 = f2_pack(f0, f0), m1 = f2_pack(f1, f1), zero = f2_pack(0.f, 0.f);
  // x mul as 128 cen(x m1) + x m0, |.| < 2^22
  auto times = [&](F32x2 x) {
    return f2_fma(f2_pack(128.f, 128.f), md.centered(f2_fma(x, m1, zero)), f2_fma(x, m0, zero));
  };
  if (!j.last) {
#pragma unroll
    for (int i = 0; i < 32; i += 2) {
      F32x2 x = md.centered(f2_pack(v[i], v[i + 1]));
      if (e.mul != 1u) x = md.centered(times(x));            // two-limb moduli
      f2_unpack(x, v[i], v[i + 1]);
    }
    tc::tmem_st32(taddr, v);
    if (e.dbg != nullptr) dbg_write_back(e.dbg, j.plane, j.u.ell, e.L1, e.M, e.N, e.row, col, taddr);
    return;
  }
  // v_l in [0, m), two to a word: one-limb |x mul| < 2^16; two-limb once more centered first
  const F32x2 up = f2_pack(8388608.0f, 8388608.0f);          // the bits of 2^23 + v end in v
#pragma unroll
  for (int i = 0; i < 32; i += 2) {
    F32x2 x = md.centered(f2_pack(v[i], v[i + 1]));
    if (two) x = md.centered(times(x));
    else x = f2_fma(x, m0, zero);
    f2_unpack(f2_add(md.floored(x), up), v[i], v[i + 1]);
    v[i >> 1] = __byte_perm(v[i], v[i + 1], 0x5410);
  }
  // staged tile: by TMA where u's rows allow it, else row by row
  const int lane = threadIdx.x & 31;
  const uint32_t buf = us.sbuf + (us.n & 1u) * 2048u;
  if (us.map != nullptr) {
    if (us.n >= 2) {                               // the buffer's previous store has read it
      if (lane == 0) tc::bulk_wait_read<1>();
      __syncwarp();
    }
  } else {
    // no TMA store may still read the buffer (a batch mixes both forms, and
    // only TMA stores count as bulk groups: wait for all of them)
    if (lane == 0) tc::bulk_wait_read<0>();
    __syncwarp();
  }
#pragma unroll
  for (int q = 0; q < 4; ++q)
    tc::st_shared_v4(buf + (uint32_t)(lane * 64 + 16 * (q ^ ((lane >> 1) & 3))), v[4 * q], v[4 * q + 1],
                     v[4 * q + 2], v[4 * q + 3]);
  ++us.n;
  if (us.map != nullptr) {
    tc::fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) {
      tc::tma_store_3d(us.map, buf, col, e.row - lane, e.ell);   // rows >= M, columns >= N are not written
      tc::bulk_commit();
    }
  } else {
    __syncwarp();
    store_tile_rows(e.uell, buf, e.row - lane, col, e.M, e.N);
  }
}

// Outputs of up to kNarrow columns take the chunks that hold any of them: the others
// cost as much as those, most of the stage for a few vectors (plane GEMMs with every
// chunk and so, ms: 4578 x 2 x 89 p = 151 0.094 and 0.035, 673 x 4 x 34 p = 1798 0.157
// and 0.057, 2000 x 60 x 500 p = 256 0.088 and 0.059).  Wider ones take all: leaving out
// the last tile's gave 1531 x 1093 x 1777 p = 512 1.13 for 1.14, but 64 uneven products
// 8.02 for 7.87.  A function of its own, so that the common loop keeps its code: eight
// 1024 x 1024 x 64 p = 512 1.436 ms, 1.453 with the bound in that loop.
constexpr int kNarrow = 128;
static __device__ __noinline__ uint32_t epi_job_narrow(Job j, EpiConst e, uint32_t tbase, UStage us, int nc) {
  uint32_t v[32];
  for (int c = 0; c < nc; ++c) {
    tc::tmem_ld32_nowait(tbase + (uint32_t)(32 * c), v);
    tc::tmem_ld_wait_regs(v);
    epi_chunk(j, e, v, tbase + (uint32_t)(32 * c), 32 * c, us);
  }
  if (!j.last) tc::tmem_wait_st();
  return us.n;
}

// The epilogue of one job over NC chunks of 32 columns at tbase, the TMEM
// load of each chunk in flight while the one before it is reduced.  Ends
// with every TMEM store of the job complete.
template <int NC>
__device__ __forceinline__ void epi_job(const Job& j, const EpiConst& e, uint32_t tbase, UStage& us) {
  static_assert(NC % 2 == 0, "chunks go in pairs");
  if (e.N <= kNarrow) {
    us.n = epi_job_narrow(j, e, tbase, us, min(NC, (e.N - e.col0 + 31) >> 5));
    return;
  }
  uint32_t va[32], vb[32];
  tc::tmem_ld32_nowait(tbase, va);
  tc::tmem_ld_wait_regs(va);
#pragma unroll 1
  for (int c = 0; c < NC; c += 2) {
    tc::tmem_ld32_nowait(tbase + (uint32_t)(32 * (c + 1)), vb);
    epi_chunk(j, e, va, tbase + (uint32_t)(32 * c), 32 * c, us);
    tc::tmem_ld_wait_regs(vb);
    if (c + 2 < NC) tc::tmem_ld32_nowait(tbase + (uint32_t)(32 * (c + 2)), va);
    epi_chunk(j, e, vb, tbase + (uint32_t)(32 * (c + 1)), 32 * (c + 1), us);
    if (c + 2 < NC) tc::tmem_ld_wait_regs(va);
  }
  if (!j.last) tc::tmem_wait_st();
}

}  // namespace plane
}  // namespace oz2
