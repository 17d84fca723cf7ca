// Fourier-domain multiply-accumulate of the operator (Sec. 3.2, Eq. 16 term (ii)):
//   forward  Y[b][t][k] = sum_z Hh[k][t][z] X[b][z][k]          (Eq. 7)
//   adjoint  Z[b][z][k] = sum_t conj(Hh[k][t][z]) D[b][t][k]    (Eq. 11)
// for every stored frequency bin k. The table is read exactly once per call,
// so both kernels are HBM-bound table streams (1 flop per table byte):
//   - a CTA owns 32 consecutive bins (one per lane); the table is stored
//     [k/32][t][z-group][lane][z in group] so every warp load is 32 x 16 B =
//     512 contiguous bytes, streamed with evict-first loads;
//   - forward: the CTA's X tile (all z of its 32 bins, VB volumes) sits in
//     shared memory; warps split the time samples and each thread produces
//     Y for one (bin, t);
//   - adjoint: warps split the z-groups, each thread keeps its Z partial sums
//     in registers while walking t; D comes through the read-only cache.
// Real tables (even kernels) store one float per (k, t, z): the real and
// imaginary parts of X are contracted by the same real coefficient.
#include <algorithm>

#include "async.cuh"
#include "pat_internal.h"

namespace pat {
namespace {

constexpr int kWarps = 8;
constexpr int64_t kFoldCtas = 304;  // two CTAs on each of 152 SMs

template <typename R, bool CPLX>
struct Elem;  // table element type and z per 16-byte group
template <> struct Elem<float, false>  { typedef float T; static constexpr int ZG = 4; };
template <> struct Elem<float, true>   { typedef cx<float> T; static constexpr int ZG = 2; };
template <> struct Elem<double, false> { typedef double T; static constexpr int ZG = 2; };
template <> struct Elem<double, true>  { typedef cx<double> T; static constexpr int ZG = 1; };

// Streamed (evict-first) 16-byte load of the table.
__device__ __forceinline__ float4 ld_stream(const float4* p) { return __ldcs(p); }
__device__ __forceinline__ double2 ld_stream(const double2* p) { return __ldcs(p); }

// Read-only-cache load of one complex value.
__device__ __forceinline__ cx<float> ldg_cx(const cx<float>* p) {
  const float2 v = __ldg(reinterpret_cast<const float2*>(p));
  return mk<float>(v.x, v.y);
}
__device__ __forceinline__ cx<double> ldg_cx(const cx<double>* p) {
  const double2 v = __ldg(reinterpret_cast<const double2*>(p));
  return mk<double>(v.x, v.y);
}

// Unpacks one 16-byte table group into ZG elements.
template <typename R, bool CPLX>
__device__ __forceinline__ void unpack(const typename vec16<R>::type& v,
                                       typename Elem<R, CPLX>::T* e);
template <> __device__ __forceinline__ void unpack<float, false>(const float4& v, float* e) {
  e[0] = v.x; e[1] = v.y; e[2] = v.z; e[3] = v.w;
}
template <> __device__ __forceinline__ void unpack<float, true>(const float4& v, cx<float>* e) {
  e[0] = mk<float>(v.x, v.y); e[1] = mk<float>(v.z, v.w);
}
template <> __device__ __forceinline__ void unpack<double, false>(const double2& v, double* e) {
  e[0] = v.x; e[1] = v.y;
}
template <> __device__ __forceinline__ void unpack<double, true>(const double2& v, cx<double>* e) {
  e[0] = mk<double>(v.x, v.y);
}

// acc += h x   (forward)   /   acc += conj(h) x   (adjoint)
template <typename R>
__device__ __forceinline__ void mac(cx<R>& acc, R h, cx<R> x) {
  acc.x = fma(h, x.x, acc.x);
  acc.y = fma(h, x.y, acc.y);
}
// Real coefficient times complex value in FP32 as one paired FMA
// (fma.rn.f32x2: each lane rounded once, as the scalar FMAs are).
__device__ __forceinline__ void mac(cx<float>& acc, float h, cx<float> x) {
  asm("{\n .reg .b64 rh, rx, ra;\n mov.b64 rh, {%2, %2};\n mov.b64 rx, {%3, %4};\n"
      " mov.b64 ra, {%0, %1};\n fma.rn.f32x2 ra, rh, rx, ra;\n mov.b64 {%0, %1}, ra;\n}"
      : "+f"(acc.x), "+f"(acc.y)
      : "f"(h), "f"(x.x), "f"(x.y));
}
template <typename R>
__device__ __forceinline__ void mac(cx<R>& acc, cx<R> h, cx<R> x) {
  acc.x = fma(h.x, x.x, acc.x);
  acc.x = fma(-h.y, x.y, acc.x);
  acc.y = fma(h.x, x.y, acc.y);
  acc.y = fma(h.y, x.x, acc.y);
}
template <typename R>
__device__ __forceinline__ void mac_conj(cx<R>& acc, R h, cx<R> x) {
  mac(acc, h, x);
}
template <typename R>
__device__ __forceinline__ void mac_conj(cx<R>& acc, cx<R> h, cx<R> x) {
  acc.x = fma(h.x, x.x, acc.x);
  acc.x = fma(h.y, x.y, acc.x);
  acc.y = fma(h.x, x.y, acc.y);
  acc.y = fma(-h.y, x.x, acc.y);
}

// grid (ceil(batch / VB), nkb): the volume groups of a block of bins are
// neighbours and share its table rows through L2. Block kWarps * 32; dynamic smem VB * nzg*ZG * 32 complex.
template <typename R, bool CPLX, int VB>
__global__ void __launch_bounds__(kWarps * 32)
    k_contract_fwd(const typename vec16<R>::type* __restrict__ table,
                   const cx<R>* __restrict__ X, cx<R>* __restrict__ Y, int nz, int nt, int nzg,
                   int64_t K, int64_t Kpad, int batch) {
  typedef typename vec16<R>::type V;
  typedef typename Elem<R, CPLX>::T E;
  constexpr int ZG = Elem<R, CPLX>::ZG;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cx<R>* xs = reinterpret_cast<cx<R>*>(smem_raw);  // [VB][nzg*ZG][32]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t kb = blockIdx.y;
  const int64_t k = kb * 32 + lane;
  const int b0 = blockIdx.x * VB;
  const int nzp = nzg * ZG;
  pdl_wait();
  for (int i = threadIdx.x; i < VB * nzp * 32; i += blockDim.x) {
    const int l = i & 31, z = (i >> 5) % nzp, v = (i >> 5) / nzp;
    const int64_t kk = kb * 32 + l;
    cx<R> a = mk<R>(0, 0);
    if (b0 + v < batch && z < nz && kk < K) a = X[((int64_t)(b0 + v) * nz + z) * Kpad + kk];
    xs[i] = a;
  }
  __syncthreads();
  const V* tb = table + (kb * nt) * (int64_t)nzg * 32 + lane;
  for (int t = warp; t < nt; t += kWarps) {
    cx<R> acc[VB];
#pragma unroll
    for (int v = 0; v < VB; ++v) acc[v] = mk<R>(0, 0);
    const V* hp = tb + (int64_t)t * nzg * 32;
#pragma unroll 4
    for (int g = 0; g < nzg; ++g) {
      E e[ZG];
      unpack<R, CPLX>(ld_stream(hp + g * 32), e);
#pragma unroll
      for (int q = 0; q < ZG; ++q) {
#pragma unroll
        for (int v = 0; v < VB; ++v) mac(acc[v], e[q], xs[(v * nzp + g * ZG + q) * 32 + lane]);
      }
    }
    if (k < K) {
#pragma unroll
      for (int v = 0; v < VB; ++v)
        if (b0 + v < batch) Y[((int64_t)(b0 + v) * nt + t) * Kpad + k] = acc[v];
    }
  }
}

// grid (ceil(batch / VB), nkb, z-chunks); block kWarps * 32. Warp w of z-chunk c
// owns the z-groups g = c * kWarps * GPW + w + j * kWarps, j < GPW. Single-
// volume float variants are held to 32 registers so 8 CTAs (all 64 warp slots)
// stay resident: the stream needs the warps more than the registers.
//
// Samples walked at a time, their loads in flight together. Complex float
// tables: eight for one volume (128^2 x 64 x 256, 4.3 GB: 716 -> 622 us, 650
// with two; 384 x 326 x 12 x 40: 217 -> 204), four for two (833 -> 675). Four for real tables with four volumes
// (128 x 96 on 256 x 192: 536 -> 422) and in FP64 with one (64^2 x 32 x 128:
// 143 -> 134); one elsewhere (single real volumes live on occupancy).
template <typename R, bool CPLX, int VB, int GPW>
__host__ __device__ constexpr int adj_unroll() {
  if (sizeof(R) == 4 && CPLX) return VB == 1 ? 8 : 4;
  if (!CPLX && GPW <= 2 && VB == (sizeof(R) == 4 ? 4 : 1)) return 4;
  return 1;
}

template <typename R, bool CPLX, int VB, int GPW>
__global__ void __launch_bounds__(kWarps * 32, (sizeof(R) == 4 && !CPLX && VB == 1 && GPW <= 2) ? 8 : 1)
    k_contract_adj(const typename vec16<R>::type* __restrict__ table,
                   const cx<R>* __restrict__ D, cx<R>* __restrict__ Z, int nz, int nt, int nzg,
                   int64_t K, int64_t Kpad, int batch) {
  typedef typename vec16<R>::type V;
  typedef typename Elem<R, CPLX>::T E;
  constexpr int ZG = Elem<R, CPLX>::ZG;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t kb = blockIdx.y;
  const int64_t k = kb * 32 + lane;
  const int b0 = blockIdx.x * VB;
  const int gbase = blockIdx.z * kWarps * GPW + warp;
  cx<R> acc[GPW][ZG][VB];
#pragma unroll
  for (int j = 0; j < GPW; ++j)
#pragma unroll
    for (int q = 0; q < ZG; ++q)
#pragma unroll
      for (int v = 0; v < VB; ++v) acc[j][q][v] = mk<R>(0, 0);
  const bool kok = k < K;
  const V* tb = table + (kb * nt) * (int64_t)nzg * 32 + lane;
  constexpr int kUnroll = adj_unroll<R, CPLX, VB, GPW>();
  pdl_wait();
#pragma unroll(kUnroll)
  for (int t = 0; t < nt; ++t) {
    cx<R> d[VB];
#pragma unroll
    for (int v = 0; v < VB; ++v)
      d[v] = (kok && b0 + v < batch) ? ldg_cx(&D[((int64_t)(b0 + v) * nt + t) * Kpad + k])
                                     : mk<R>(0, 0);
    const V* hp = tb + (int64_t)t * nzg * 32;
#pragma unroll
    for (int j = 0; j < GPW; ++j) {
      const int g = gbase + j * kWarps;
      if (g < nzg) {
        E e[ZG];
        unpack<R, CPLX>(ld_stream(hp + g * 32), e);
#pragma unroll
        for (int q = 0; q < ZG; ++q)
#pragma unroll
          for (int v = 0; v < VB; ++v) mac_conj(acc[j][q][v], e[q], d[v]);
      }
    }
  }
  if (!kok) return;
#pragma unroll
  for (int j = 0; j < GPW; ++j) {
    const int g = gbase + j * kWarps;
#pragma unroll
    for (int q = 0; q < ZG; ++q) {
      const int z = g * ZG + q;
      if (g < nzg && z < nz) {
#pragma unroll
        for (int v = 0; v < VB; ++v)
          if (b0 + v < batch) Z[((int64_t)(b0 + v) * nz + z) * Kpad + k] = acc[j][q][v];
      }
    }
  }
}

// ---- D4-folded real tables ----------------------------------------------------
// A CTA owns 32 representatives {|kx|, |ky|} (one per lane); the table row of
// a representative is read once and applied to each of its (up to 4) bins,
// whose bin indices come from `members` ([block][lane][4], -1 = absent). CTA j
// reads stored chunk chunk[j] of 32 rows (chunk j when `chunk` is NULL): with
// radial sharing the CTAs of one radius group read the same chunk at about
// the same time, so DRAM delivers it once and L2 serves the others; the
// volumes of a batch are neighbouring CTAs for the same reason.
//
// The members of a block's representatives are scattered over the half
// spectrum, so with one row of bins per slice every access is an 8-byte piece
// of a 32-byte sector. GRP spectra interleave eight slices ([slice / 8][bin]
// [slice % 8], see SpecRow): a lane's eight time samples (depths) of one bin
// are 64 contiguous bytes, two whole sectors. The spectra of a block are
// staged in shared memory in quads of four slices, [member][quad][lane] with
// the 16-byte halves of a quad swizzled so that a warp's 16-byte reads touch
// every bank once.
//
// Measured per launch (one GB300, forward / adjoint): 128^2 -> 256^2 x 64 x
// 256, 0.40 GB stored: 87 / 88 us, from 110 / 113 with bin rows and the table
// loaded into registers; 256^2 -> 512^2 x 128 x 512, 5.8 GB: 1170 / 1176 from
// 2270 / 1915; 202^2 -> 512^2 x 17 x 201: 119 / 147 from 507 / 316; five
// volumes at 64^2 -> 128^2 x 32 x 128: 32 / 38 from 57 / 76. What bounds them
// is the load / store unit: a block of 4 samples reads its spectra (32 cycles
// a step and warp), the ring (16), stages and stores scattered sectors (a cycle
// per line): 64 us of the 87 at 128^2, beside 62 us of DRAM traffic and 34 us
// of multiply-adds.
constexpr int kFoldThreads = 512;  // most threads of a CTA (caps the registers at 128)

// 16-byte slot of half h (slices 2h, 2h + 1) of a lane's quad in its 1 KB row.
__device__ __forceinline__ int quad_slot(int lane, int h) {
  return (2 * lane + h) ^ ((lane >> 2) & 1);
}

// Offset of quad q (slices 4q .. 4q + 3) of a bin in grouped spectra.
__device__ __forceinline__ int64_t group_off(int q, int64_t bin, int64_t Kpad) {
  return ((int64_t)(q >> 1) * Kpad + bin) * kGroup + (q & 1) * 4;
}

// Starts the copy of quads [q0, q0 + nq) of the four members' spectra into
// dst[4][rows][64] (16-byte slots); slices at or past n and absent members
// become zero. in: this volume's spectra.
template <bool GRP>
__device__ __forceinline__ void stage_quads(float4* dst, int rows, const cx<float>* in,
                                            const int* bins, int q0, int nq, int n, int64_t Kpad,
                                            int lane, int warp, int nwarps) {
  for (int q = warp; q < nq; q += nwarps) {
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const bool ok = bins[m] >= 0;
      const int64_t bin = ok ? bins[m] : 0;
      float4* row = dst + (m * rows + q) * 64;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint32_t d = (uint32_t)__cvta_generic_to_shared(row + quad_slot(lane, h));
        const int s = 4 * (q0 + q) + 2 * h;  // first slice of this half
        if constexpr (GRP) {
          const int bytes = ok ? 8 * max(0, min(2, n - s)) : 0;
          const cx<float>* src = in + group_off(q0 + q, bin, Kpad) + 2 * h;
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d),
                       "l"(bytes ? src : in), "r"(bytes)
                       : "memory");
        } else {
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int bytes = ok && s + i < n ? 8 : 0;
            const cx<float>* src = in + (int64_t)(s + i) * Kpad + bin;
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d + 8 * i),
                         "l"(bytes ? src : in), "r"(bytes)
                         : "memory");
          }
        }
      }
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// Stores the values of four consecutive slices 4q .. 4q + 3 of one bin.
template <bool GRP>
__device__ __forceinline__ void store_quad(cx<float>* out, int q, int bin, int n, int64_t Kpad,
                                           cx<float> a, cx<float> b, cx<float> c, cx<float> d) {
  if constexpr (GRP) {  // slices at or past n are padding that no reader uses
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(
                     out + group_off(q, bin, Kpad)),
                 "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y), "f"(d.x), "f"(d.y)
                 : "memory");
  } else {
    cx<float>* o = out + (int64_t)(4 * q) * Kpad + bin;
    if (4 * q < n) o[0] = a;
    if (4 * q + 1 < n) o[Kpad] = b;
    if (4 * q + 2 < n) o[2 * Kpad] = c;
    if (4 * q + 3 < n) o[3 * Kpad] = d;
  }
}

// Stores quad q of the four members, v[slice of the quad][member]. In rows
// (GRP false) a frequency shard's members are four consecutive aligned slots:
// one 32-byte store per slice then takes the place of four scattered 8-byte
// ones.
template <bool GRP>
__device__ __forceinline__ void store_members(cx<float>* out, int q, const int* bins, int n,
                                              int64_t Kpad, const cx<float> (*v)[4]) {
  if constexpr (!GRP) {
    cx<float>* o = out + (int64_t)(4 * q) * Kpad + bins[0];
    const bool run = bins[0] >= 0 && bins[1] == bins[0] + 1 && bins[2] == bins[0] + 2 &&
                     bins[3] == bins[0] + 3;
    if (run && ((reinterpret_cast<uintptr_t>(o) | (uintptr_t)(Kpad * 8)) & 31) == 0) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (4 * q + i < n)
          asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(
                           o + i * Kpad),
                       "f"(v[i][0].x), "f"(v[i][0].y), "f"(v[i][1].x), "f"(v[i][1].y),
                       "f"(v[i][2].x), "f"(v[i][2].y), "f"(v[i][3].x), "f"(v[i][3].y)
                       : "memory");
      return;
    }
  }
#pragma unroll
  for (int m = 0; m < 4; ++m)
    if (bins[m] >= 0)
      store_quad<GRP>(out, q, bins[m], n, Kpad, v[0][m], v[1][m], v[2][m], v[3][m]);
}

// Adds what store_quad wrote to a .. d.
template <bool GRP>
__device__ __forceinline__ void add_quad(const cx<float>* out, int q, int bin, int n, int64_t Kpad,
                                         cx<float>& a, cx<float>& b, cx<float>& c, cx<float>& d) {
  const cx<float>* o = GRP ? out + group_off(q, bin, Kpad) : out + (int64_t)(4 * q) * Kpad + bin;
  const int64_t st = GRP ? 1 : Kpad;
  a = cadd(a, o[0]);
  if (4 * q + 1 < n) b = cadd(b, o[st]);
  if (4 * q + 2 < n) c = cadd(c, o[2 * st]);
  if (4 * q + 3 < n) d = cadd(d, o[3 * st]);
}

// Complex values per volume of a spectrum of n slices.
template <bool GRP>
__device__ __forceinline__ int64_t vol_len(int n, int64_t Kpad) {
  return (GRP ? (int64_t)((n + kGroup - 1) / kGroup) * kGroup : (int64_t)n) * Kpad;
}

template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// A warp's ring of R slots of SLOT float4 rows (32 lanes) in shared memory,
// filled by bulk copies of contiguous pieces of the table: lane 0 issues the
// copies of a step, all lanes wait for it and read their own column, and the
// slot is refilled as soon as every lane has read it, so R steps are in flight
// and their bytes cost neither registers nor load / store slots. A wait tests
// its barrier `limit` times at most. Once one runs out on any lane the ring is
// dead for the whole warp: nothing more is issued, read or passed, so slot, par
// and fly go on naming every copy in flight (the step waited for among them),
// and close() waits for these before the warp leaves its shared memory.
template <int R, int SLOT>
struct TableRing {
  float4* rows;    // [R][SLOT][32]
  uint64_t* full;  // [R]
  uint32_t limit;
  int slot = 0;    // of the oldest step: the one to read, and then to refill
  uint32_t par = 0;
  int fly = 0;     // steps issued and not read
  bool dead = false;
  __device__ __forceinline__ TableRing(unsigned char* smem, uint64_t* bars, int warp, int lane,
                                       uint32_t lim)
      : rows(reinterpret_cast<float4*>(smem) + warp * (R * SLOT * 32)),
        full(bars + warp * R),
        limit(lim) {
    if (lane == 0) {
      for (int i = 0; i < R; ++i) mbar_init(&full[i], 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
  }
  // Opens slot i for copies of `bytes` in all (lane 0). The lanes' reads of the
  // slot, ordinary loads before a __syncwarp, come before the copies that
  // overwrite it: different proxies, so a fence. It costs what the loads still
  // in flight take (forward / adjoint 83 / 89 us without, 87 / 88 with it at
  // 128^2 x 64 x 256; 1154 / 1154 and 1225 / 1165 at 256^2 x 128 x 512, both in
  // blocks of 4). Later in the step it costs more: the copies then start late.
  __device__ __forceinline__ float4* open(int i, uint32_t bytes) {
    fence_proxy_async();
    mbar_arrive_expect_tx(&full[i], bytes);
    return rows + i * (SLOT * 32);
  }
  __device__ __forceinline__ void copy(int i, float4* dst, const float4* src, int nrows) {
    bulk_g2s(dst, src, (uint32_t)nrows * 512u, &full[i]);
  }
  // Waits for the oldest step, its slot in `src`; false, on every lane, once the
  // ring is dead.
  __device__ __forceinline__ bool wait(const float4** src) {
    dead = !__all_sync(0xffffffffu, mbar_wait(&full[slot], par, limit));
    *src = rows + slot * (SLOT * 32);
    return !dead;
  }
  // The oldest step has been read by this warp and its slot refilled.
  __device__ __forceinline__ void next() {
    if (++slot == R) {
      slot = 0;
      par ^= 1u;
    }
  }
  // Every lane of a dead ring's warp leaves once lane 0 has seen the copies land
  // (kDrainNs at most).
  __device__ __forceinline__ void close(int lane, int* err) {
    if (!dead) return;
    if (lane == 0) {
      atomicExch(err, 1);
      const uint64_t deadline = global_ns() + kDrainNs;
      for (; fly > 0; --fly, next()) drain_wait(&full[slot], par, deadline);
    }
    __syncwarp();
  }
};

// Warp index, uniform for the compiler: the cursors of the rings then live in
// uniform registers.
__device__ __forceinline__ int warp_index() {
  return __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);
}

// Forward: a warp takes blocks of T time samples and walks the z-groups, a
// step of its ring holding the T table rows of one group; tb time blocks per
// split. grid (batch, nrb, splits of the time blocks): the volumes of a block
// share its table rows through L2. Rows: (splits, nrb, batch), since their
// scattered 8-byte pieces are gathered into lines in L2 while one volume is
// worked on (three volumes at 100^2 x 33 x 201: 329 us interleaved, 209 in turn).
template <bool GRP, int T, int R>
__global__ void __launch_bounds__(kFoldThreads, 1)
    k_fold_fwd(const float4* __restrict__ table, const int4* __restrict__ members,
               const int* __restrict__ chunk, const cx<float>* __restrict__ X,
               cx<float>* __restrict__ Y, int nz, int nt, int nzg, int64_t Kpad, int tb, int gc,
               uint32_t limit, int* __restrict__ err) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = warp_index(), nwarps = blockDim.x >> 5;
  float4* xs = reinterpret_cast<float4*>(smem_raw);  // [4][gc][64]
  unsigned char* rings = smem_raw + 4096 * gc;
  TableRing<R, T> ring(rings, reinterpret_cast<uint64_t*>(rings + nwarps * (R * T * 512)), warp,
                       lane, limit);
  const int64_t ub = blockIdx.y;
  const int b = GRP ? blockIdx.x : blockIdx.z, split = GRP ? blockIdx.z : blockIdx.x;
  const float4* tbl = table + (int64_t)(chunk ? chunk[ub] : ub) * nt * nzg * 32;
  const int bk0 = split * tb + warp;
  const int bend = min((nt + T - 1) / T, (split + 1) * tb);
  for (int g0 = 0; g0 < nzg; g0 += gc) {  // z-groups whose spectra fit: one pass up to gc groups
    const int g1 = min(nzg, g0 + gc);
    int pbk = bk0, pg = g0;  // next step to copy
    auto refill = [&](int i) {
      if (pbk < bend && !ring.dead) {
        if (lane == 0) {
          const int n = min(T, nt - pbk * T);
          float4* dst = ring.open(i, (uint32_t)n * 512u);
#pragma unroll
          for (int r = 0; r < T; r += 4)
            if (r < n)
              ring.copy(i, dst + r * 32, tbl + folded_row(pbk * T + r, pg, nt, nzg),
                        min(4, n - r));
        }
        ++ring.fly;
        if (++pg == g1) {
          pg = g0;
          pbk += nwarps;
        }
      }
    };
#pragma unroll
    for (int i = 0; i < R; ++i) refill((ring.slot + i) % R);  // the table is constant: no wait
    {
      const int4 mem = members[ub * 32 + lane];
      const int bins[4] = {mem.x, mem.y, mem.z, mem.w};
      if (g0 == 0) pdl_wait();
      stage_quads<GRP>(xs, gc, X + b * vol_len<GRP>(nz, Kpad), bins, g0, g1 - g0, nz, Kpad, lane,
                       warp, nwarps);
    }
    cp_wait<0>();
    __syncthreads();
    for (int bk = bk0; bk < bend && !ring.dead; bk += nwarps) {
      cx<float> acc[T][4];
#pragma unroll
      for (int r = 0; r < T; ++r)
#pragma unroll
        for (int m = 0; m < 4; ++m) acc[r][m] = mk<float>(0.f, 0.f);
#pragma unroll 1
      for (int g = 0; g < g1 - g0; ++g) {
        const float4* hs;
        if (!ring.wait(&hs)) break;
        float4 h[T];
#pragma unroll
        for (int r = 0; r < T; ++r) h[r] = hs[r * 32 + lane];
        --ring.fly;
        __syncwarp();
        refill(ring.slot);
        ring.next();
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          float4 x[4];
#pragma unroll
          for (int m = 0; m < 4; ++m) x[m] = xs[(m * gc + g) * 64 + quad_slot(lane, hf)];
#pragma unroll
          for (int r = 0; r < T; ++r)
#pragma unroll
            for (int m = 0; m < 4; ++m) {
              mac(acc[r][m], hf ? h[r].z : h[r].x, mk<float>(x[m].x, x[m].y));
              mac(acc[r][m], hf ? h[r].w : h[r].y, mk<float>(x[m].z, x[m].w));
            }
        }
      }
      if (ring.dead) break;
      const int4 mem = __ldg(members + ub * 32 + lane);
      const int bins[4] = {mem.x, mem.y, mem.z, mem.w};
      cx<float>* Yb = Y + b * vol_len<GRP>(nt, Kpad);
#pragma unroll
      for (int r = 0; r < T; r += 4) {
        const int q = (bk * T + r) / 4;
        if (4 * q >= nt) break;
        if (g0 > 0) {
#pragma unroll
          for (int m = 0; m < 4; ++m)
            if (bins[m] >= 0)
              add_quad<GRP>(Yb, q, bins[m], nt, Kpad, acc[r][m], acc[r + 1][m], acc[r + 2][m],
                            acc[r + 3][m]);
        }
        store_members<GRP>(Yb, q, bins, nt, Kpad, &acc[r]);
      }
    }
    if (g1 < nzg) __syncthreads();  // the spectra are free
  }
  ring.close(lane, err);
}

// Forward on rows, table rows through registers. What bounds it is the scattered
// 8-byte accesses to the spectra; without rings two CTAs an SM leave the L1 that
// gathers them 100 KB. Blocks of 4 samples, every depth resident. 128^2 x 64 x
// 256: 100 us, 114 through rings; 100^2 x 33 x 201: 59 and 90; on one frequency
// shard 89 and 96, 48 and 58. grid (1, nrb, batch).
__global__ void __launch_bounds__(kWarps * 32, 2)
    k_fold_fwd_rows(const float4* __restrict__ table, const int4* __restrict__ members,
                    const int* __restrict__ chunk, const cx<float>* __restrict__ X,
                    cx<float>* __restrict__ Y, int nz, int nt, int nzg, int64_t Kpad) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cx<float>* xs = reinterpret_cast<cx<float>*>(smem_raw);  // [4][nzp][32]
  const int lane = threadIdx.x & 31, warp = warp_index(), nzp = nzg * 4;
  const int64_t ub = blockIdx.y;
  const int4 mem = members[ub * 32 + lane];
  const int bins[4] = {mem.x, mem.y, mem.z, mem.w};
  const cx<float>* Xb = X + (int64_t)blockIdx.z * nz * Kpad;
  cx<float>* Yb = Y + (int64_t)blockIdx.z * nt * Kpad;
  pdl_wait();
  for (int z = warp; z < nzp; z += kWarps) {
#pragma unroll
    for (int m = 0; m < 4; ++m)
      xs[(m * nzp + z) * 32 + lane] =
          bins[m] >= 0 && z < nz ? Xb[(int64_t)z * Kpad + bins[m]] : mk<float>(0.f, 0.f);
  }
  __syncthreads();
  const float4* tbl = table + (int64_t)(chunk ? chunk[ub] : ub) * nt * nzg * 32 + lane;
  for (int t0 = 4 * warp; t0 < nt; t0 += 4 * kWarps) {
    cx<float> acc[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int m = 0; m < 4; ++m) acc[r][m] = mk<float>(0.f, 0.f);
    const int n = min(4, nt - t0);
    const float4* hp = tbl + folded_row(t0, 0, nt, nzg);
#pragma unroll 4
    for (int g = 0; g < nzg; ++g) {
      float4 h[4];
#pragma unroll
      for (int r = 0; r < 4; ++r)
        h[r] = r < n ? ld_stream(hp + (g * n + r) * 32) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        cx<float> x[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) x[m] = xs[(m * nzp + g * 4 + q) * 32 + lane];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const float hq = q == 0 ? h[r].x : q == 1 ? h[r].y : q == 2 ? h[r].z : h[r].w;
#pragma unroll
          for (int m = 0; m < 4; ++m) mac(acc[r][m], hq, x[m]);
        }
      }
    }
    store_members<false>(Yb, t0 / 4, bins, nt, Kpad, acc);
  }
}

// Adjoint: warp (zi, ti) of zw x tw owns the z-groups (zc zw + zi) GPW + j
// (j < GPW) and the quads ti, ti + tw, ...; the 4 members' D of SQ tw quads
// are staged in shared memory (two buffers, the next stage's copies in flight
// during the current one) and reused by all warps; the table comes through
// the warp's ring as in the forward. With tw > 1 the warps' partial sums of
// one z-group meet in shared memory at the end, in the order of ti. grid
// (z-chunks x batch, nrb), rows (z-chunks, nrb, batch) as in the forward.
template <bool GRP, int GPW, int SQ, int R>
__global__ void __launch_bounds__(kFoldThreads, 1)
    k_fold_adj(const float4* __restrict__ table, const int4* __restrict__ members,
               const int* __restrict__ chunk, const cx<float>* __restrict__ D,
               cx<float>* __restrict__ Z, int nz, int nt, int nzg, int64_t Kpad, int nzc, int zw,
               int tw, uint32_t limit, int* __restrict__ err) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = warp_index(), nwarps = blockDim.x >> 5;
  const int tq = SQ * tw;                            // quads per stage
  float4* ds = reinterpret_cast<float4*>(smem_raw);  // [2][4][tq][64]
  unsigned char* rings = smem_raw + 2 * 4096 * tq;
  TableRing<R, 4 * GPW> ring(
      rings, reinterpret_cast<uint64_t*>(rings + nwarps * (R * 4 * GPW * 512)), warp, lane,
      limit);
  const int64_t ub = blockIdx.y;
  const int zc = GRP ? blockIdx.x % nzc : blockIdx.x, b = GRP ? blockIdx.x / nzc : blockIdx.z;
  const int zi = warp % zw, ti = warp / zw;
  const int gbase = (zc * zw + zi) * GPW;
  const float4* tbl = table + (int64_t)(chunk ? chunk[ub] : ub) * nt * nzg * 32;
  const int ntq = (nt + 3) / 4, nst = (ntq + tq - 1) / tq;
  int pq = gbase < nzg ? ti : ntq;  // next quad to copy
  auto refill = [&](int i) {
    if (pq < ntq && !ring.dead) {
      if (lane == 0) {
        const int n = min(4, nt - 4 * pq), ng = min(GPW, nzg - gbase);
        float4* dst = ring.open(i, (uint32_t)(n * ng) * 512u);
#pragma unroll
        for (int j = 0; j < GPW; ++j)
          if (j < ng) ring.copy(i, dst + j * 128, tbl + folded_row(4 * pq, gbase + j, nt, nzg), n);
      }
      ++ring.fly;
      pq += tw;
    }
  };
#pragma unroll
  for (int i = 0; i < R; ++i) refill(i);
  const int4 mem = members[ub * 32 + lane];
  const int bins[4] = {mem.x, mem.y, mem.z, mem.w};
  const cx<float>* Db = D + b * vol_len<GRP>(nt, Kpad);
  cx<float> acc[GPW][4][4];
#pragma unroll
  for (int j = 0; j < GPW; ++j)
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int m = 0; m < 4; ++m) acc[j][q][m] = mk<float>(0.f, 0.f);
  pdl_wait();
  stage_quads<GRP>(ds, tq, Db, bins, 0, min(tq, ntq), nt, Kpad, lane, warp, nwarps);
  for (int st = 0; st < nst; ++st) {
    const int q0 = st * tq;
    cp_wait<0>();     // this stage's D
    __syncthreads();  // and every warp is done with the other buffer
    if (st + 1 < nst)
      stage_quads<GRP>(ds + ((st + 1) & 1) * 4 * tq * 64, tq, Db, bins, q0 + tq,
                       min(tq, ntq - q0 - tq), nt, Kpad, lane, warp, nwarps);
    const float4* dst = ds + (st & 1) * 4 * tq * 64;
#pragma unroll 1
    for (int q = ti; q < min(tq, ntq - q0) && gbase < nzg && !ring.dead; q += tw) {
      const float4* hs;
      if (!ring.wait(&hs)) break;
      float4 h[4][GPW];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int j = 0; j < GPW; ++j) h[r][j] = hs[(j * 4 + r) * 32 + lane];
      float4 d0[4];  // read before the fence of the refill holds lane 0 up
#pragma unroll
      for (int m = 0; m < 4; ++m) d0[m] = dst[(m * tq + q) * 64 + quad_slot(lane, 0)];
      --ring.fly;
      __syncwarp();
      refill(ring.slot);
      ring.next();
      if (4 * (q0 + q) + 4 > nt) {  // rows past nt were not copied; D is zero there
#pragma unroll
        for (int r = 1; r < 4; ++r)
#pragma unroll
          for (int j = 0; j < GPW; ++j)
            if (4 * (q0 + q) + r >= nt) h[r][j] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int hf = 0; hf < 2; ++hf)
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const float4 d = hf ? dst[(m * tq + q) * 64 + quad_slot(lane, 1)] : d0[m];
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const cx<float> dv = k ? mk<float>(d.z, d.w) : mk<float>(d.x, d.y);
#pragma unroll
            for (int j = 0; j < GPW; ++j) {
              const float4 hv = h[2 * hf + k][j];
              mac(acc[j][0][m], hv.x, dv);
              mac(acc[j][1][m], hv.y, dv);
              mac(acc[j][2][m], hv.z, dv);
              mac(acc[j][3][m], hv.w, dv);
            }
          }
        }
    }
  }
  ring.close(lane, err);
  if (tw > 1) {
    __syncthreads();  // the staging buffers and rings are free
    cx<float>* red = reinterpret_cast<cx<float>*>(smem_raw);  // [(ti - 1) zw + zi][GPW 16][32]
    if (ti > 0) {
      cx<float>* r = red + ((ti - 1) * zw + zi) * (GPW * 16 * 32) + lane;
#pragma unroll
      for (int j = 0; j < GPW; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int m = 0; m < 4; ++m) r[((j * 4 + q) * 4 + m) * 32] = acc[j][q][m];
    }
    __syncthreads();
    if (ti == 0)
      for (int k = 1; k < tw; ++k) {
        const cx<float>* r = red + ((k - 1) * zw + zi) * (GPW * 16 * 32) + lane;
#pragma unroll
        for (int j = 0; j < GPW; ++j)
#pragma unroll
          for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int m = 0; m < 4; ++m)
              acc[j][q][m] = cadd(acc[j][q][m], r[((j * 4 + q) * 4 + m) * 32]);
      }
  }
  if (ti != 0) return;
  cx<float>* Zb = Z + b * vol_len<GRP>(nz, Kpad);
#pragma unroll
  for (int j = 0; j < GPW; ++j) {
    const int g = gbase + j;
    if (g >= nzg) break;
#pragma unroll
    for (int m = 0; m < 4; ++m)
      if (bins[m] >= 0)
        store_quad<GRP>(Zb, g, bins[m], nz, Kpad, acc[j][0][m], acc[j][1][m], acc[j][2][m],
                        acc[j][3][m]);
  }
}

// Adjoint on rows, table rows through registers: warp w of a z-chunk owns the
// z-groups w and w + 8 of 16; the members' D of 32 samples at a time in shared
// memory, the loads of 8 samples in flight together. Bound as k_fold_fwd_rows.
// 128^2 x 128 x 128: 111 us, 134 through rings; 128^2 x 112 x 64 60 and 72, on one
// frequency shard 50 and 68. grid (z-chunks, nrb, batch).
__global__ void __launch_bounds__(kWarps * 32, 2)
    k_fold_adj_rows(const float4* __restrict__ table, const int4* __restrict__ members,
                    const int* __restrict__ chunk, const cx<float>* __restrict__ D,
                    cx<float>* __restrict__ Z, int nz, int nt, int nzg, int64_t Kpad) {
  constexpr int GPW = 2, TC = 32;
  __shared__ cx<float> ds[TC][4][32];
  const int lane = threadIdx.x & 31, warp = warp_index();
  const int64_t ub = blockIdx.y;
  const int4 mem = members[ub * 32 + lane];
  const int bins[4] = {mem.x, mem.y, mem.z, mem.w};
  const int gbase = blockIdx.x * kWarps * GPW + warp;
  const cx<float>* Db = D + (int64_t)blockIdx.z * nt * Kpad;
  const float4* tbl = table + (int64_t)(chunk ? chunk[ub] : ub) * nt * nzg * 32 + lane;
  cx<float> acc[GPW][4][4];
#pragma unroll
  for (int j = 0; j < GPW; ++j)
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int m = 0; m < 4; ++m) acc[j][q][m] = mk<float>(0.f, 0.f);
  pdl_wait();
  for (int t0 = 0; t0 < nt; t0 += TC) {
    __syncthreads();
    for (int tt = warp; tt < TC; tt += kWarps) {
#pragma unroll
      for (int m = 0; m < 4; ++m)
        ds[tt][m][lane] = bins[m] >= 0 && t0 + tt < nt ? Db[(int64_t)(t0 + tt) * Kpad + bins[m]]
                                                       : mk<float>(0.f, 0.f);
    }
    __syncthreads();
    const int tn = min(TC, nt - t0);
    for (int tt = 0; tt < tn; tt += 8) {
      float4 h[8][GPW];
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int j = 0; j < GPW; ++j) {
          const int g = gbase + j * kWarps;
          h[r][j] = g < nzg && tt + r < tn ? ld_stream(tbl + folded_row(t0 + tt + r, g, nt, nzg))
                                           : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        cx<float> d[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) d[m] = ds[(tt + r) & (TC - 1)][m][lane];
#pragma unroll
        for (int j = 0; j < GPW; ++j) {
          const float hq[4] = {h[r][j].x, h[r][j].y, h[r][j].z, h[r][j].w};
#pragma unroll
          for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int m = 0; m < 4; ++m) mac(acc[j][q][m], hq[q], d[m]);
        }
      }
    }
  }
#pragma unroll
  for (int j = 0; j < GPW; ++j) {
    const int g = gbase + j * kWarps;
    if (g >= nzg) break;
    store_members<false>(Z + (int64_t)blockIdx.z * nz * Kpad, g, bins, nz, Kpad, acc[j]);
  }
}

constexpr size_t kSmemCta = 227 * 1024;  // most shared memory of a CTA (and of an SM's CTAs)

// one: one CTA of up to 16 warps per SM even where two would fit.
template <bool GRP, int T, int R>
cudaError_t fold_fwd_t(const Plan& p, const void* X, void* Y, int batch, int gc, bool one,
                       cudaStream_t s) {
  const Layout& L = p.L;
  constexpr size_t ring = (size_t)R * (T * 512 + 8);  // bytes per warp
  const size_t xbytes = (size_t)gc * 4096;
  const bool two = !one && 2 * (xbytes + 8 * ring) <= kSmemCta;
  const int nwarps = two ? 8 : (int)std::min<size_t>(16, (kSmemCta - xbytes) / ring);
  const size_t smem = xbytes + nwarps * ring;
  auto fn = k_fold_fwd<GRP, T, R>;
  cudaError_t e = allow_smem(fn, smem);
  if (e != cudaSuccess) return e;
  // Splits of the time blocks over CTAs, by waves of CTAs x (blocks of the
  // busiest warp + the CTA's load of its SM + its prologue): the order of the
  // measured times at 71 to 1059 blocks (64^2: 9.2 us in 2, 14.5 in 1; 128^2:
  // 83 us in 1, 91 in 2; 5 volumes at 64^2: 31 us in 2, 33.5 in 1; all without
  // the fence of a refill).
  const int nb = (L.nt + T - 1) / T, slots = two ? (int)kFoldCtas : (int)kFoldCtas / 2;
  const int64_t ctas = L.nrb * batch;
  int tb = nb;
  double best = 1e300;
  for (int split = 1; split <= 8; split *= 2) {
    const int n = (nb + split - 1) / split, parts = (nb + n - 1) / n;
    const double cost = (double)((ctas * parts + slots - 1) / slots) *
                        ((n + nwarps - 1) / nwarps + 0.1 * n + 0.5);
    if (cost < best) {
      best = cost;
      tb = n;
    }
  }
  const unsigned splits = (unsigned)((nb + tb - 1) / tb);
  const dim3 grid(GRP ? (unsigned)batch : splits, (unsigned)L.nrb, GRP ? splits : (unsigned)batch);
  return launch_pdl(fn, grid, dim3(nwarps * 32), smem, s, static_cast<const float4*>(p.table),
                    reinterpret_cast<const int4*>(p.rb_members),
                    static_cast<const int*>(p.rb_chunk), static_cast<const cx<float>*>(X),
                    static_cast<cx<float>*>(Y), L.nz, L.nt, L.nzg, L.Kpad, tb, gc,
                    (uint32_t)p.tc_spin, p.tc_err);
}

cudaError_t fold_fwd(const Plan& p, const void* X, void* Y, int batch, bool grouped,
                     cudaStream_t s) {
  const Layout& L = p.L;
  if ((size_t)L.nzg * 4096 > kSmemCta) return cudaErrorInvalidValue;  // more than 224 depths
  // the spectra of up to 128 depths are resident at a time, more take another pass
  const int gc = std::min(L.nzg, 32);
  const int64_t ctas = L.nrb * batch;
  if (!grouped) {
    // Rows, in bins or in a shard's slots. Up to a CTA per SM: rings of 16 warps,
    // the time samples split (64^2 x 32 x 128: 12.1 us, 13.0 in CTAs of 8 warps,
    // 18.7 without rings; one shard of four of 128^2 x 64 x 256: 31, 36, 58).
    // More CTAs hide the table's latency themselves: no rings (see
    // k_fold_fwd_rows). Slots are stored in 32-byte runs, which leaves the rings
    // ahead at few depths (17 on 404^2: 140 us and 155) and past 112, where the
    // spectra leave room for one CTA (128^2 x 128 x 128: 107 and 120).
    if (ctas <= kFoldCtas / 2) return fold_fwd_t<false, 4, 2>(p, X, Y, batch, gc, true, s);
    if (p.shard_world && L.nzg > 28) return fold_fwd_t<false, 8, 1>(p, X, Y, batch, gc, false, s);
    if (p.shard_world && L.nzg <= 5) return fold_fwd_t<false, 4, 2>(p, X, Y, batch, gc, false, s);
    const size_t smem = (size_t)L.nzg * 4096;
    const cudaError_t e = allow_smem(k_fold_fwd_rows, smem);
    if (e != cudaSuccess) return e;
    return launch_pdl(k_fold_fwd_rows, dim3(1, (unsigned)L.nrb, (unsigned)batch), dim3(kWarps * 32),
                      smem, s, static_cast<const float4*>(p.table),
                      reinterpret_cast<const int4*>(p.rb_members),
                      static_cast<const int*>(p.rb_chunk), static_cast<const cx<float>*>(X),
                      static_cast<cx<float>*>(Y), L.nz, L.nt, L.nzg, L.Kpad);
  }
  // Blocks of 8 samples read the spectra half as often as blocks of 4 and take
  // half as many fences (TableRing::open). With two steps in the ring two CTAs
  // fit an SM up to 48 depths (three volumes at 96^2 x 45: 75 us, 81 in blocks
  // of 4). Beyond, blocks of 8 have one step in the ring, which pays from two
  // waves of CTAs on: two CTAs an SM up to 80 depths (128^2 x 64: 89 us in
  // blocks of 4 with three steps, 91 in blocks of 8; five volumes 402 and 351),
  // then one of 16 warps (256^2 x 128 x 512: 1212 and 1165; 71 CTAs at
  // 64^2 x 128 x 256: 47 and 50). Blocks of 4 with three steps fit two CTAs an SM
  // up to 64 depths; from 65 to 80 two with two steps are ahead once they fill
  // three quarters of the SMs' places (128^2 x 80 x 200, 277 CTAs: 93 us, 106 in
  // one CTA of 16 warps with three; 213 CTAs of 64^2 x 80 x 100: 47 and 41).
  const size_t xbytes = (size_t)gc * 4096;
  if (2 * (xbytes + 8 * 2 * (8 * 512 + 8)) <= kSmemCta)
    return fold_fwd_t<true, 8, 2>(p, X, Y, batch, gc, false, s);
  if (ctas >= 2 * kFoldCtas) return fold_fwd_t<true, 8, 1>(p, X, Y, batch, gc, false, s);
  if (L.nzg > 16 && L.nzg <= 20 && 4 * ctas > 3 * kFoldCtas)
    return fold_fwd_t<true, 4, 2>(p, X, Y, batch, gc, false, s);
  return fold_fwd_t<true, 4, 3>(p, X, Y, batch, gc, false, s);
}

template <bool GRP, int GPW, int SQ, int R>
cudaError_t fold_adj_t(const Plan& p, const void* D, void* Z, int batch, int zw, int tw,
                       cudaStream_t s) {
  const Layout& L = p.L;
  const int nzc = (L.nzg + zw * GPW - 1) / (zw * GPW), nwarps = zw * tw;
  const size_t ring = (size_t)nwarps * R * (4 * GPW * 512 + 8);
  const size_t smem = std::max<size_t>(2 * 4096 * (size_t)SQ * tw + ring,
                                       (size_t)(tw - 1) * zw * GPW * 4096);
  auto fn = k_fold_adj<GRP, GPW, SQ, R>;
  cudaError_t e = allow_smem(fn, smem);
  if (e != cudaSuccess) return e;
  const dim3 grid((unsigned)(GRP ? nzc * batch : nzc), (unsigned)L.nrb, GRP ? 1u : (unsigned)batch);
  return launch_pdl(fn, grid, dim3(nwarps * 32), smem, s, static_cast<const float4*>(p.table),
                    reinterpret_cast<const int4*>(p.rb_members),
                    static_cast<const int*>(p.rb_chunk), static_cast<const cx<float>*>(D),
                    static_cast<cx<float>*>(Z), L.nz, L.nt, L.nzg, L.Kpad, nzc, zw, tw,
                    (uint32_t)p.tc_spin, p.tc_err);
}

// Two z-groups per warp and up to 8 warps along z; fewer along z leave warps
// for the time samples. Grids with less than about one CTA per SM split the
// z-groups over more CTAs (64^2 x 32: 12.1 us in two, 16 in one; 32^2 x 16:
// 5.8 us in four of one group per warp, 13 in one). A stage holds two quads of
// D per warp along the time, or four from two waves of CTAs on (256^2 x 128 x
// 512: 1175 us with two, 1154 with four; five volumes at 128^2 346 and 332; so
// far without the fence of a refill). In
// rows a stage of one leaves L1 more room to gather bins (100^2 x 33 x 201: 64 us,
// 76 with two, 123 with four; one shard of 128^2 x 32 x 128 36, 48, 50), but for a
// shard from 64 depths on (64^2 x 128 x 256: 72 with one, 63 with two). With more
// CTAs than SMs, 64 depths or more and few samples rows take no rings
// (k_fold_adj_rows; 100^2 x 64 x 64 33 us, 38 through rings, one shard of 256^2 x
// 64 x 128 227 and 241; but 128^2 x 64 x 256 107 and 105, five volumes of it 543
// and 494, one shard of 256^2 x 128 x 512 1452 and 1327).
template <bool GRP>
cudaError_t fold_adj(const Plan& p, const void* D, void* Z, int batch, cudaStream_t s) {
  const Layout& L = p.L;
  const int64_t ctas = L.nrb * batch;
  if (!GRP && ctas > kFoldCtas / 2 && L.nzg >= 16 && L.nt <= (L.nzg > 16 ? 256 : 128))
    return launch_pdl(k_fold_adj_rows,
                      dim3((unsigned)((L.nzg + 15) / 16), (unsigned)L.nrb, (unsigned)batch),
                      dim3(kWarps * 32), 0, s, static_cast<const float4*>(p.table),
                      reinterpret_cast<const int4*>(p.rb_members),
                      static_cast<const int*>(p.rb_chunk), static_cast<const cx<float>*>(D),
                      static_cast<cx<float>*>(Z), L.nz, L.nt, L.nzg, L.Kpad);
  const int units = (L.nzg + 1) / 2;
  int nzc = (units + 7) / 8;
  int zw = (units + nzc - 1) / nzc;
  while (zw > 1 && 2 * ctas * nzc <= 200) {
    zw = (zw + 1) / 2;
    nzc = (units + zw - 1) / zw;
  }
  if (zw == 1 && 2 * ctas * nzc <= 200) return fold_adj_t<GRP, 1, 1, 4>(p, D, Z, batch, 1, 8, s);
  static constexpr int kTw[8] = {8, 4, 2, 2, 1, 1, 1, 1};
  const int tw = kTw[zw - 1];
  if constexpr (GRP) {
    if (tw == 1 && ctas * nzc >= 2 * kFoldCtas)
      return fold_adj_t<GRP, 2, 4, 2>(p, D, Z, batch, zw, tw, s);
  }
  return tw <= 2 && (GRP || (p.shard_world && L.nzg >= 16))
             ? fold_adj_t<GRP, 2, 2, 2>(p, D, Z, batch, zw, tw, s)
             : fold_adj_t<GRP, 2, 1, 2>(p, D, Z, batch, zw, tw, s);
}

template <typename R, bool CPLX, int VB>
cudaError_t fwd_t(const Plan& p, const void* X, void* Y, int batch, cudaStream_t s) {
  const Layout& L = p.L;
  constexpr int ZG = Elem<R, CPLX>::ZG;
  const size_t smem = sizeof(cx<R>) * (size_t)VB * L.nzg * ZG * 32;
  auto fn = k_contract_fwd<R, CPLX, VB>;
  const cudaError_t e = allow_smem(fn, smem);
  if (e != cudaSuccess) return e;
  dim3 grid((unsigned)((batch + VB - 1) / VB), (unsigned)L.nkb);
  return launch_pdl(fn, grid, dim3(kWarps * 32), smem, s,
                    static_cast<const typename vec16<R>::type*>(p.table),
                    static_cast<const cx<R>*>(X), static_cast<cx<R>*>(Y), L.nz, L.nt, L.nzg, L.K,
                    L.Kpad, batch);
}

template <typename R, bool CPLX, int VB, int GPW>
cudaError_t adj_launch(const Plan& p, const void* D, void* Z, int batch, cudaStream_t s) {
  const Layout& L = p.L;
  const int per_chunk = kWarps * GPW;
  dim3 grid((unsigned)((batch + VB - 1) / VB), (unsigned)L.nkb,
            (unsigned)((L.nzg + per_chunk - 1) / per_chunk));
  return launch_pdl(k_contract_adj<R, CPLX, VB, GPW>, grid, dim3(kWarps * 32), 0, s,
                    static_cast<const typename vec16<R>::type*>(p.table),
                    static_cast<const cx<R>*>(D), static_cast<cx<R>*>(Z), L.nz, L.nt, L.nzg, L.K,
                    L.Kpad, batch);
}

template <typename R, bool CPLX, int VB>
cudaError_t adj_t(const Plan& p, const void* D, void* Z, int batch, cudaStream_t s) {
  // z-groups per warp: enough to cover nzg in one chunk up to 4 per warp,
  // beyond that several z-chunks each re-read D (small) but not the table.
  const int nzg = p.L.nzg;
  if constexpr (sizeof(R) == 8) {
    // The FP64 rate bounds these, and their time follows the slots for groups,
    // those at or past nzg included: the fewest slots, then the fewest chunks.
    // 17 groups (34 depths, 128 samples) in 32 slots and in 24: 128^2 1026 and
    // 711 us, 64^2 303 and 210; complex, 34 groups in 64 and in 40: 574 and 337.
    auto slots = [&](int gpw) { return (nzg + kWarps * gpw - 1) / (kWarps * gpw) * gpw; };
    if (slots(1) < std::min(slots(2), slots(4))) return adj_launch<R, CPLX, VB, 1>(p, D, Z, batch, s);
    if (slots(2) < slots(4)) return adj_launch<R, CPLX, VB, 2>(p, D, Z, batch, s);
    return adj_launch<R, CPLX, VB, 4>(p, D, Z, batch, s);
  }
  if (nzg <= kWarps) return adj_launch<R, CPLX, VB, 1>(p, D, Z, batch, s);
  if (nzg <= 2 * kWarps) return adj_launch<R, CPLX, VB, 2>(p, D, Z, batch, s);
  return adj_launch<R, CPLX, VB, 4>(p, D, Z, batch, s);
}

// Volumes per table pass: a group of VB volumes reads the table once; the
// groups of a block of bins are neighbouring CTAs, which share it through L2.
template <typename R, bool CPLX>
cudaError_t fwd_vb(const Plan& p, const void* X, void* Y, int batch, cudaStream_t s) {
  // as many volumes as their spectra leave room for
  const size_t one = sizeof(cx<R>) * (size_t)p.L.nzg * Elem<R, CPLX>::ZG * 32;
  if (batch >= 4 && 4 * one <= kSmemCta) return fwd_t<R, CPLX, 4>(p, X, Y, batch, s);
  if (batch >= 2 && 2 * one <= kSmemCta) return fwd_t<R, CPLX, 2>(p, X, Y, batch, s);
  return fwd_t<R, CPLX, 1>(p, X, Y, batch, s);
}
template <typename R, bool CPLX>
cudaError_t adj_vb(const Plan& p, const void* D, void* Z, int batch, cudaStream_t s) {
  // complex float tables in pairs: four volumes' D in one CTA push the table
  // out of L1 (2085 us a launch at 128^2 x 64 x 256), two groups of two read
  // the same rows through L2 (1049 us)
  if constexpr (!(CPLX && sizeof(R) == 4))
    if (batch >= 4) return adj_t<R, CPLX, 4>(p, D, Z, batch, s);
  if (batch >= 2) return adj_t<R, CPLX, 2>(p, D, Z, batch, s);
  return adj_t<R, CPLX, 1>(p, D, Z, batch, s);
}

}  // namespace

// Rows [volumes][n][Kpad] <-> grouped slices: a thread holds the eight slices
// of one bin, a warp reads or writes 256 bytes of a row at a time. Bound by the
// bytes. The padding bins K .. Kpad of either side are left alone.
template <bool TO>
__global__ void __launch_bounds__(256) k_regroup(const float2* __restrict__ in,
                                                 float2* __restrict__ out, int n, int G,
                                                 int64_t K, int64_t Kpad, int kblocks) {
  const int vg = blockIdx.x / kblocks, v = vg / G, g = vg - v * G;
  const int64_t k = (int64_t)(blockIdx.x - vg * kblocks) * 256 + threadIdx.x;
  if (k >= K) return;
  const int left = n - g * kGroup;  // slices of this group, eight or more but in the last
  const int64_t row = ((int64_t)v * n + g * kGroup) * Kpad + k;
  const int64_t grp = ((int64_t)vg * Kpad + k) * kGroup;
  float2 x[kGroup];
  pdl_wait();
  if constexpr (TO) {
#pragma unroll
    for (int j = 0; j < kGroup; ++j)
      x[j] = j < left ? in[row + j * Kpad] : make_float2(0.f, 0.f);
    float4* o = reinterpret_cast<float4*>(out + grp);
#pragma unroll
    for (int j = 0; j < kGroup / 2; ++j)
      o[j] = make_float4(x[2 * j].x, x[2 * j].y, x[2 * j + 1].x, x[2 * j + 1].y);
  } else {
    const float4* src = reinterpret_cast<const float4*>(in + grp);
#pragma unroll
    for (int j = 0; j < kGroup / 2; ++j) {
      const float4 q = src[j];
      x[2 * j] = make_float2(q.x, q.y);
      x[2 * j + 1] = make_float2(q.z, q.w);
    }
#pragma unroll
    for (int j = 0; j < kGroup; ++j)
      if (j < left) out[row + j * Kpad] = x[j];
  }
}

template <bool TO>
cudaError_t regroup(const Plan& p, const void* in, void* out, int volumes, int n, cudaStream_t s) {
  const int G = (n + kGroup - 1) / kGroup, kblocks = (int)((p.L.K + 255) / 256);
  const int64_t blocks = (int64_t)volumes * G * kblocks;
  if (blocks > 0x7fffffff) return cudaErrorInvalidValue;
  return launch_pdl(k_regroup<TO>, dim3((unsigned)blocks), dim3(256), 0, s,
                    static_cast<const float2*>(in), static_cast<float2*>(out), n, G, p.L.K,
                    p.L.Kpad, kblocks);
}

cudaError_t launch_to_groups(const Plan& p, const void* in, void* out, int volumes, int n,
                             cudaStream_t s) {
  return regroup<true>(p, in, out, volumes, n, s);
}

cudaError_t launch_from_groups(const Plan& p, const void* in, void* out, int volumes, int n,
                               cudaStream_t s) {
  return regroup<false>(p, in, out, volumes, n, s);
}

cudaError_t launch_contract_fwd(const Plan& p, const void* X, void* Y, int batch, cudaStream_t s,
                                bool grouped) {
  if (p.tc_fwd && p.tc_min_batch > 0 && batch >= p.tc_min_batch)
    return tc_contract(p, p.tc_fwd, p.tc_adj, X, Y, batch, false, p.tc_err, s, grouped);
  if (p.L.fold) return fold_fwd(p, X, Y, batch, grouped, s);
  if (p.L.fp64)
    return p.L.real ? fwd_vb<double, false>(p, X, Y, batch, s) : fwd_vb<double, true>(p, X, Y, batch, s);
  return p.L.real ? fwd_vb<float, false>(p, X, Y, batch, s) : fwd_vb<float, true>(p, X, Y, batch, s);
}

cudaError_t launch_contract_adj(const Plan& p, const void* D, void* Z, int batch, cudaStream_t s,
                                bool grouped) {
  if (p.tc_adj && p.tc_min_batch > 0 && batch >= p.tc_min_batch)
    return tc_contract(p, p.tc_fwd, p.tc_adj, D, Z, batch, true, p.tc_err, s, grouped);
  if (p.L.fold) return grouped ? fold_adj<true>(p, D, Z, batch, s) : fold_adj<false>(p, D, Z, batch, s);
  if (p.L.fp64)
    return p.L.real ? adj_vb<double, false>(p, D, Z, batch, s) : adj_vb<double, true>(p, D, Z, batch, s);
  return p.L.real ? adj_vb<float, false>(p, D, Z, batch, s) : adj_vb<float, true>(p, D, Z, batch, s);
}

}  // namespace pat
