// Device code for the two-component Shan-Chen D3Q19 evaporation step
// (arXiv:1701.03637, Sec. II) shared by all launches of the library.
//
// State between launches ("pre-stream" form): the buffer holds post-collision
// populations f*(t-1). One launch pulls them (streaming with halfway
// bounce-back), applies the evaporation sink to the arrived populations, forms
// densities and Psi, the Eq. (3) force, and collides (Eqs. (1), (2) with the
// tau F / rho velocity shift), writing f*(t) to the other buffer. The canonical
// (post-stream, post-sink) populations of step t are pull + sink of the buffer.
//
// Memory layout: 19 arrays (one per direction) of np pairs (r, b): the populations of both
// components in one word (float2, or two 16-bit values), so that a load, a store and a copy
// move both (with an array per component, half the instructions of a pull were address
// arithmetic and copies: 256^3 FP16 step 0.90 -> 0.80 ms, 151 x 93 x 67 FP32 90 -> 69 us);
// site s = x + nx (y + ny z) with x fastest, rows contiguous without padding so
// that neighbouring tiles share every fetched sector through L2. Periodic wrap
// is index arithmetic.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

namespace sclbm {

constexpr int Q = 19;
constexpr int FLUID = 0, SINK = 1, SOLID = 2;
constexpr int kGhosts = 2;  // copied planes on each side of a shifted lattice

// D3Q19, own order: rest, +-x, +-y, +-z, then the 12 face diagonals in
// opposite pairs (i odd, i+1) with e_{i+1} = -e_i.
__host__ __device__ constexpr int dir_x(int i) {
  return (i == 1 || i == 7 || i == 9 || i == 11 || i == 13) ? 1
       : (i == 2 || i == 8 || i == 10 || i == 12 || i == 14) ? -1 : 0;
}
__host__ __device__ constexpr int dir_y(int i) {
  return (i == 3 || i == 7 || i == 10 || i == 15 || i == 17) ? 1
       : (i == 4 || i == 8 || i == 9 || i == 16 || i == 18) ? -1 : 0;
}
__host__ __device__ constexpr int dir_z(int i) {
  return (i == 5 || i == 11 || i == 14 || i == 15 || i == 18) ? 1
       : (i == 6 || i == 12 || i == 13 || i == 16 || i == 17) ? -1 : 0;
}
__host__ __device__ constexpr int opp(int i) { return i == 0 ? 0 : ((i & 1) ? i + 1 : i - 1); }
// e_y + 1 and e_z + 1 of all 19 directions in 2 bits each, for runtime direction indices.
constexpr unsigned long long pack_dir(int axis) {
  unsigned long long v = 0;
  for (int i = 0; i < 19; ++i)
    v |= (unsigned long long)((axis == 1 ? dir_y(i) : dir_z(i)) + 1) << (2 * i);
  return v;
}
constexpr unsigned long long kDirY = pack_dir(1), kDirZ = pack_dir(2);
__device__ __forceinline__ int dir_y_rt(int i) { return (int)((kDirY >> (2 * i)) & 3ull) - 1; }
__device__ __forceinline__ int dir_z_rt(int i) { return (int)((kDirZ >> (2 * i)) & 3ull) - 1; }
// Lattice weights (Sec. II A): 1/3 rest, 1/18 axis, 1/36 diagonal. In FP32 they are
// chosen within two ulps of those values so that w0 + 6 w1 + 12 w2 == 1 exactly:
// with the nearest floats the sum is 1 + 2^-26 and every collision would create
// that fraction of its mass (a steady drift of the conserved totals).
constexpr float kW1 = 14913080.0f * 0x1p-28f;  // 1/18 - 1 ulp
constexpr float kW2 = 7456540.0f * 0x1p-28f;   // kW1 / 2 exactly
constexpr float kW0 = 11184812.0f * 0x1p-25f;  // 1 - 12 kW1 exactly
__host__ __device__ constexpr float wgt(int i) { return i == 0 ? kW0 : (i <= 6 ? kW1 : kW2); }
__host__ __device__ constexpr double wgt_d(int i) { return i == 0 ? 1.0 / 3.0 : (i <= 6 ? 1.0 / 18.0 : 1.0 / 36.0); }

// ------------------------------------------------------------------ pair arithmetic
// Both components of a site go through the same operations, so the kernels hold them as
// pairs V = float2 (r, b) and issue one packed instruction (add / mul / fma .f32x2) for
// the two: the same correctly rounded result in each half as the scalar operation, half
// the instructions. V = float runs one component (an odd component of the N-component step).
__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
// The compiler contracts a packed sum of a packed product that has no other use, written with
// the builtins or in PTX, also as fma(c, 1, a b) (20.7% of 8.4M random a b + c differed from the
// scalar operations); a sum or difference through fma by -1 is kept, and so is a product that a sum
// and a difference share (none differed). So no product goes into vadd alone: vsub is the fma by
// -1, relax_core's odd part is both added and subtracted, and StF16S decodes with scalar products.
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// a - b = (-1) b + a, rounded once
__device__ __forceinline__ float2 vsub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }
__device__ __forceinline__ float vneg(float a) { return -a; }
__device__ __forceinline__ float2 vneg(float2 a) { return make_float2(-a.x, -a.y); }
template <class V>
__device__ __forceinline__ V vset(float a);
template <>
__device__ __forceinline__ float vset<float>(float a) { return a; }
template <>
__device__ __forceinline__ float2 vset<float2>(float a) { return make_float2(a, a); }

// Everything a launch needs to know about one lattice.
struct LatDev {
  int nx, ny, nz, nxny;
  long long np;            // pairs between consecutive direction arrays (N components: populations)
  float omega[2], tau[2];  // 1/tau and tau per component
  float G, rhoH;           // g of Eq. (3); imposed rho^r at sinks
  float Gs[2];             // self couplings g^{rr}, g^{bb} of Eq. (3) (0: the paper's two-component model)
  double rhoH_mass;        // exact sum of the reset r populations fl(w_i rho_H)
  int geometry, sink_z0, sink_layers;  // sink_z0 in [0, nz)
  double scx, scy, scz, RH2;
  float sc32[3], RH2_32, r2_tol;       // the sphere in FP32, and the error bound of FP32 r^2 - RH2
  int wall_z0, wall_z1;    // solid slab [wall_z0, wall_z1)
  // z-slab of a larger lattice: local plane z is plane (z + zoff) mod nzg of the lattice
  // whose geometry (sinks, walls, sphere) these fields describe; planes [own0, own1) are
  // the slab's own, the rest ghosts whose evaporation is not booked. A whole lattice has
  // zoff = 0, nzg = nz, own0 = 0, own1 = nz.
  int zoff, nzg, own0, own1;
};

// Plane of the whole lattice that local plane z is (z in [0, nz)).
__device__ __forceinline__ int global_z(const LatDev& L, int z) {
  int g = z + L.zoff;
  g = g >= L.nzg ? g - L.nzg : g;
  return g >= L.nzg ? g - L.nzg : g;
}
__device__ __forceinline__ bool own_z(const LatDev& L, int z) { return z >= L.own0 && z < L.own1; }

// ------------------------------------------------------------------ storage types
// Asynchronous copy of a pair (4 or 8 bytes), cached in L1.
template <int BYTES>
__device__ __forceinline__ void cp_async_ca(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(sa), "l"(gmem), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// Bulk copies (the TMA engine) into shared memory, completing on an mbarrier.
__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned arrivals) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(arrivals) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
__device__ __forceinline__ void mbar_expect(uint64_t* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Waits until the phase of the given parity completes; false when it has not within 2 s.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, unsigned parity) {
  if (mbar_try(bar, parity)) return true;
  const unsigned long long t0 = global_ns();
  while (!mbar_try(bar, parity))
    if (global_ns() - t0 > 2000000000ull) return false;
  return true;
}
// A box of the tensor at element coordinates (x, y, z, i); the x start must lie on a
// 16-byte boundary, parts outside the tensor are filled with zeros.
__device__ __forceinline__ void tma_load4(void* smem, const CUtensorMap* map, int x, int y, int z, int i, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
      "[%6];\n" ::"r"(smem_addr(smem)),
      "l"(map), "r"(x), "r"(y), "r"(z), "r"(i), "r"(smem_addr(bar))
      : "memory");
}
// 16-byte asynchronous copy, cached in L2 only; both addresses 16-byte aligned.
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(smem)), "l"(gmem) : "memory");
}

// T: the stored pair (r, b) of one direction; cv decodes it and enc encodes it (w is the
// direction's weight), each half with the single population's operations. ld, ldcg: a pair
// from global memory, ldcg at L2 only (never from L1), for kernels in which other CTAs of the
// same launch overwrite the data between two reads. put: population stores to global memory
// are evict-first: the next step reads them only after the whole lattice has gone by, and until
// then they can displace what neighbouring CTAs share in the L2. The difference is small since the
// CTAs claim their work in order: evict-first / plain, us per step, shifted FP16 512 x 288 x 201 1752 /
// 1765, FP32 256^3 with the spherical sink 969 / 967, 512^3 6889 / 6873.
struct StF32 {
  using T = float2;
  static __device__ __forceinline__ float2 cv(T v, float) { return v; }
  static __device__ __forceinline__ T enc(float2 v, float) { return v; }
};
// FP16 / BF16 offsets h = f - w_i * rho0 (rho0 = 1), round to nearest even; component r in
// the low half.
__device__ __forceinline__ float2 half_pair(uint32_t v) {
  return make_float2(__half2float(__ushort_as_half((unsigned short)(v & 0xffffu))),
                     __half2float(__ushort_as_half((unsigned short)(v >> 16))));
}
__device__ __forceinline__ uint32_t half_word(float2 v) {
  const __half2 p = __floats2half2_rn(v.x, v.y);
  return (uint32_t)__half_as_ushort(__low2half(p)) | (uint32_t)__half_as_ushort(__high2half(p)) << 16;
}
struct StF16 {
  using T = uint32_t;
  static __device__ __forceinline__ float2 cv(T v, float w) { return vadd(make_float2(w, w), half_pair(v)); }
  static __device__ __forceinline__ T enc(float2 v, float w) { return half_word(vsub(v, make_float2(w, w))); }
};
// FP16 of the population scaled by its weight, g = f_i / w_i (about rho),
// round to nearest even: the same relative spacing in the liquid and the vapour.
struct StF16S {
  using T = uint32_t;
  // not a packed product: that was contracted into momentum's differences
  static __device__ __forceinline__ float2 cv(T v, float w) {
    const float2 h = half_pair(v);
    return make_float2(__fmul_rn(w, h.x), __fmul_rn(w, h.y));
  }
  // w is a compile-time weight at every call, so 1 / w folds to a constant
  static __device__ __forceinline__ T enc(float2 v, float w) { return half_word(vmul(v, make_float2(1.0f / w, 1.0f / w))); }
};
struct StBF16 {
  using T = uint32_t;
  static __device__ __forceinline__ float2 cv(T v, float w) {  // a bfloat16 is the upper half of its float
    return vadd(make_float2(w, w), make_float2(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u)));
  }
  static __device__ __forceinline__ T enc(float2 v, float w) {
    const float2 h = vsub(v, make_float2(w, w));
    const __nv_bfloat162 p = __floats2bfloat162_rn(h.x, h.y);
    return (uint32_t)__bfloat16_as_ushort(__low2bfloat16(p)) | (uint32_t)__bfloat16_as_ushort(__high2bfloat16(p)) << 16;
  }
};
template <class S>
__device__ __forceinline__ float2 ld(const typename S::T* p, float w) { return S::cv(__ldg(p), w); }
template <class S>
__device__ __forceinline__ float2 ldcg(const typename S::T* p, float w) { return S::cv(__ldcg(p), w); }
template <class S>
__device__ __forceinline__ void put(typename S::T* p, float2 v, float w) { __stcs(p, S::enc(v, w)); }

__host__ __device__ __forceinline__ int wrapi(int v, int n) {
  v %= n;
  return v < 0 ? v + n : v;
}
// Periodic wrap without a division when v is within one period of [0, n).
__host__ __device__ __forceinline__ int wrap_near(int v, int n) {
  v = v < 0 ? v + n : (v >= n ? v - n : v);
  return (unsigned)v < (unsigned)n ? v : wrapi(v, n);
}

__device__ __forceinline__ bool solid_z(const LatDev& L, int z) {
  const int g = global_z(L, z);
  return g >= L.wall_z0 && g < L.wall_z1;
}

// Site class from coordinates (no storage): solid slab, planar or spherical sink.
// The squared distance is formed without FMA contraction so it rounds like a
// plain host evaluation. z is a local plane; the geometry is the whole lattice's.
__device__ __forceinline__ int site_class(const LatDev& L, int x, int y, int zl) {
  if (solid_z(L, zl)) return SOLID;
  const int z = global_z(L, zl);
  if (L.geometry == 1) {
    const int dz = z - L.sink_z0;  // sink_z0 in [0, nzg), z in [0, nzg)
    return (dz < 0 ? dz + L.nzg : dz) < L.sink_layers ? SINK : FLUID;
  }
  if (L.geometry == 2) {
    // FP32 first: only sites within the error bound of the sphere (72 u X^2 + u RH2, X the
    // largest extent or centre coordinate, u = 2^-24; a shell 0.01 sites thick at 256^3)
    // need the FP64 distance, which runs at 1/64 of the FP32 rate (256^3 step with the
    // sphere: 1.32 ms with FP64 at every site and halo site, 0.99 ms)
    const float fx = (float)x - L.sc32[0], fy = (float)y - L.sc32[1], fz = (float)z - L.sc32[2];
    const float far = fx * fx + fy * fy + fz * fz - L.RH2_32;
    if (fabsf(far) > L.r2_tol) return far > 0.0f ? SINK : FLUID;
    const double dx = (double)x - L.scx, dy = (double)y - L.scy, dz = (double)z - L.scz;
    const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
    return r2 >= L.RH2 ? SINK : FLUID;
  }
  return FLUID;
}

template <int I, int N>
struct Unroll {
  template <class F>
  static __device__ __forceinline__ void run(F&& f) {
    f(std::integral_constant<int, I>());
    Unroll<I + 1, N>::run(f);
  }
};
template <int N>
struct Unroll<N, N> {
  template <class F>
  static __device__ __forceinline__ void run(F&&) {}
};

// Source offsets of the pull for site (x, y, z): the population arriving in
// direction i comes from x - e_i (periodic); from a solid site it is the site's
// own opposite population (halfway bounce-back).
struct PullIdx {
  int xs[3], ys[3], zs[3];  // indexed by 1 + e (source = x - e)
  bool sol_m, sol_p;        // source plane z - 1 / z + 1 is solid
  int s;
  __device__ __forceinline__ PullIdx(const LatDev& L, int x, int y, int z) {
    const int xm = x == 0 ? L.nx - 1 : x - 1, xp = x == L.nx - 1 ? 0 : x + 1;
    const int ym = y == 0 ? L.ny - 1 : y - 1, yp = y == L.ny - 1 ? 0 : y + 1;
    const int zm = z == 0 ? L.nz - 1 : z - 1, zp = z == L.nz - 1 ? 0 : z + 1;
    xs[0] = xp; xs[1] = x; xs[2] = xm;
    ys[0] = yp * L.nx; ys[1] = y * L.nx; ys[2] = ym * L.nx;
    zs[0] = zp * L.nxny; zs[1] = z * L.nxny; zs[2] = zm * L.nxny;
    sol_p = solid_z(L, zp);
    sol_m = solid_z(L, zm);
    s = x + ys[1] + zs[1];
  }
  template <int I>
  __device__ __forceinline__ void at(int& idx, int& d) const {
    constexpr int ex = dir_x(I), ey = dir_y(I), ez = dir_z(I);
    const bool sol = ez > 0 ? sol_m : (ez < 0 ? sol_p : false);
    idx = sol ? s : xs[1 + ex] + ys[1 + ey] + zs[1 + ez];
    d = sol ? opp(I) : I;
  }
};

template <class S>
__device__ __forceinline__ void pull_full(const LatDev& L, const typename S::T* __restrict__ src, const PullIdx& P,
                                          float2 (&f)[Q]) {
  Unroll<0, Q>::run([&](auto ic) {
    constexpr int I = decltype(ic)::value;
    int idx, d;
    P.template at<I>(idx, d);
    f[I] = ld<S>(src + (long long)d * L.np + idx, wgt(I));
  });
}

// Asynchronous form of pull_full: the pair of direction i goes to sm[i stride].
template <class S>
__device__ __forceinline__ void pull_async(const LatDev& L, const typename S::T* __restrict__ src, const PullIdx& P,
                                           typename S::T* sm, int stride) {
  Unroll<0, Q>::run([&](auto ic) {
    constexpr int I = decltype(ic)::value;
    int idx, d;
    P.template at<I>(idx, d);
    cp_async_ca<sizeof(typename S::T)>(sm + I * stride, src + (long long)d * L.np + idx);
  });
}

// Density from the 19 populations of a site: opposite pairs (I, I+1) first, then
// a balanced tree (depth 5, so the additions overlap), in one fixed order that
// every kernel uses; get(i) yields population i (a float or a pair), so values can be
// summed as they are loaded.
template <class V, class Get>
__device__ __forceinline__ V sum19_of(Get&& get) {
  auto pair = [&](auto ic) {
    constexpr int I = 1 + 2 * decltype(ic)::value;
    return vadd(get(std::integral_constant<int, I>()), get(std::integral_constant<int, I + 1>()));
  };
  using std::integral_constant;
  const V c0 = vadd(pair(integral_constant<int, 0>()), pair(integral_constant<int, 1>()));
  const V c1 = vadd(pair(integral_constant<int, 2>()), pair(integral_constant<int, 3>()));
  const V c2 = vadd(pair(integral_constant<int, 4>()), pair(integral_constant<int, 5>()));
  const V c3 = vadd(pair(integral_constant<int, 6>()), pair(integral_constant<int, 7>()));
  const V c4 = vadd(pair(integral_constant<int, 8>()), get(integral_constant<int, 0>()));
  return vadd(vadd(vadd(c0, c1), vadd(c2, c3)), c4);
}
template <class V>
__device__ __forceinline__ V sum19(const V (&f)[Q]) {
  return sum19_of<V>([&](auto ic) { return f[decltype(ic)::value]; });
}

// Evaporation boundary (Sec. II C) on the densities of the arrived populations:
// rho^r := rho_H, rho^b := rho^r + rho^b - rho_H.
__device__ __forceinline__ void sink_densities(const LatDev& L, float2& rho) {
  rho.y = __fsub_rn(__fadd_rn(rho.x, rho.y), L.rhoH);
  rho.x = L.rhoH;
}

// Reset value of direction i for density rho (f^eq at rest), an exact float product.
template <class V>
__device__ __forceinline__ V rest_pop(int i, V rho) { return vmul(vset<V>(wgt(i)), rho); }

// Evaporated mass of one sink site: sum_i (f_i^r - w_i rho_H) over the arrived r
// populations, without contraction, so that where only reset values arrived (inside
// the sink region) every term is exactly zero and no rounding bias is booked.
__device__ __forceinline__ float sink_excess(const LatDev& L, const float2 (&f)[Q]) {
  float e = 0.0f;
#pragma unroll
  for (int i = 0; i < Q; ++i) e = __fadd_rn(e, __fsub_rn(f[i].x, rest_pop(i, L.rhoH)));
  return e;
}

// Eq. (4) with rho0 = 1. Below rho = 2^-6, 1 - exp(-rho) would cancel, so Psi
// is its Taylor series rho (1 - rho/2 (1 - rho/3 (1 - rho/4))) there (relative
// truncation below rho^4 / 120 <= 5e-10): trace densities keep Psi ~ rho.
__device__ __forceinline__ float psi_of(float rho) {
  if (rho < 0.015625f) {
    const float t = __fmaf_rn(-0.25f * rho, 1.0f / 3.0f, 1.0f / 3.0f);  // (1 - rho/4) / 3
    const float u = __fmaf_rn(-rho * 0.5f, t, 0.5f);                     // (1 - rho/3 (...)) / 2
    return __fmul_rn(rho, __fmaf_rn(-rho, u, 1.0f));
  }
  return 1.0f - expf(-rho);
}
__device__ __forceinline__ float2 psi_of(float2 rho) { return make_float2(psi_of(rho.x), psi_of(rho.y)); }

template <class S>
__device__ __forceinline__ void store_site(const LatDev& L, typename S::T* __restrict__ dst, int s,
                                           const float2 (&f)[Q]) {
#pragma unroll
  for (int i = 0; i < Q; ++i) put<S>(dst + (long long)i * L.np + s, f[i], wgt(i));
}

// Momentum sum_i f_i e_i of each component from the differences of opposite
// pairs, d = f_I - f_{I+1} (e_{I+1} = -e_I): each axis sums the five d whose
// e_I has a component along it.
template <class V>
__device__ __forceinline__ void momentum(const V (&f)[Q], V (&m)[3]) {
  V d[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) d[k] = vsub(f[1 + 2 * k], f[2 + 2 * k]);
  bool first[3] = {true, true, true};
  Unroll<0, 9>::run([&](auto kc) {
    constexpr int K = decltype(kc)::value, I = 1 + 2 * K;
    constexpr int e[3] = {dir_x(I), dir_y(I), dir_z(I)};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if (e[a] == 0) continue;
      if (first[a]) m[a] = e[a] > 0 ? d[K] : vneg(d[K]);
      else m[a] = e[a] > 0 ? vadd(m[a], d[K]) : vsub(m[a], d[K]);
      first[a] = false;
    }
  });
}

// The collision arithmetic below spells out every rounding (vmul, vfma, ...) so that the compiler cannot contract it differently in different kernels:
// every step kernel produces the same bits for the same state.

// Common velocity u' = sum_c (m^c / tau_c) / sum_c (rho^c / tau_c) (Sec. II A: the
// mass-weighted u_eq when tau_r = tau_b).
__device__ __forceinline__ void common_velocity(const LatDev& L, float2 rho, const float2 (&m)[3], float (&up)[3]) {
  const float omr = L.omega[0], omb = L.omega[1];
  const float den = __fmaf_rn(rho.x, omr, __fmul_rn(rho.y, omb));
  const float inv = den > 0.0f ? __fdiv_rn(1.0f, den) : 0.0f;
#pragma unroll
  for (int d = 0; d < 3; ++d) up[d] = __fmul_rn(__fmaf_rn(m[d].x, omr, __fmul_rn(m[d].y, omb)), inv);
}

// c . u for a D3Q19 direction, summing the non-zero terms in x, y, z order.
template <int I, class V>
__device__ __forceinline__ V cdot(const V (&u)[3]) {
  constexpr int ex = dir_x(I), ey = dir_y(I), ez = dir_z(I);
  V r = vset<V>(0.0f);
  bool first = true;
  if (ex != 0) { r = ex > 0 ? u[0] : vneg(u[0]); first = false; }
  if (ey != 0) { r = first ? (ey > 0 ? u[1] : vneg(u[1])) : (ey > 0 ? vadd(r, u[1]) : vsub(r, u[1])); first = false; }
  if (ez != 0) { r = first ? (ez > 0 ? u[2] : vneg(u[2])) : (ez > 0 ? vadd(r, u[2]) : vsub(r, u[2])); }
  return r;
}

// -g tau Psi / rho, the factor of A in the velocity shift (relax_core).
__device__ __forceinline__ float shift_factor(float g, float tau, float rho, float ps) {
  const float q = rho > 0.0f ? __fdiv_rn(ps, rho) : 0.0f;
  return __fmul_rn(__fmul_rn(-g, tau), q);
}
__device__ __forceinline__ float2 shift_factor(float2 g, float2 tau, float2 rho, float2 ps) {
  return make_float2(shift_factor(g.x, tau.x, rho.x, ps.x), shift_factor(g.y, tau.y, rho.y, ps.y));
}

// Shifted-velocity BGK relaxation of a component (V = float) or of both (float2) at a
// fluid site (Eqs. (1)-(3)): u_eq = u' + tau_c F^c / rho^c with F^c = -Psi^c(x) g A: g = G
// and A = a^cbar = sum_i w_i Psi^cbar(x + e_i) e_i in the paper's two-component model,
// g = 1 and A = sum_cbar g^{c cbar} a^cbar with self couplings.
template <class V>
__device__ __forceinline__ void relax_core(V om, V tau, V (&f)[Q], V rho, V ps, V g, const V (&A)[3],
                                           const float (&up)[3]) {
  // tau F / rho = (-g tau) (Psi / rho) A with Psi / rho <= 1, so a trace (or
  // denormal) density cannot overflow the shift; rho = 0 takes u' itself
  const V gq = shift_factor(g, tau, rho, ps);
  V u[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) u[d] = vfma(gq, A[d], vset<V>(up[d]));
  const V usq = vfma(u[0], u[0], vfma(u[1], u[1], vmul(u[2], u[2])));
  const V base = vfma(vset<V>(-1.5f), usq, vset<V>(1.0f));  // 1 - 1.5 u.u
  // f^eq_i = w_i rho (1 + 3 c.u + 4.5 (c.u)^2 - 1.5 u.u); opposite directions share
  // the even part w rho (1 - 1.5 u.u) + 4.5 w rho (c.u)^2 and differ in the sign of
  // the odd part 3 w rho c.u. The factors of w rho are formed once per weight class.
  f[0] = vfma(om, vsub(vmul(vmul(vset<V>(kW0), rho), base), f[0]), f[0]);
  const V wr1 = vmul(vset<V>(kW1), rho), wr2 = vmul(vset<V>(kW2), rho);
  const V wb1 = vmul(wr1, base), wb2 = vmul(wr2, base);
  const V w451 = vmul(vset<V>(4.5f), wr1), w452 = vmul(vset<V>(4.5f), wr2);
  const V w31 = vmul(vset<V>(3.0f), wr1), w32 = vmul(vset<V>(3.0f), wr2);
  Unroll<0, 9>::run([&](auto kc) {
    constexpr int I = 1 + 2 * decltype(kc)::value, J = I + 1;
    constexpr bool axis = I <= 6;
    const V cu = cdot<I>(u);
    const V ev = vfma(vmul(axis ? w451 : w452, cu), cu, axis ? wb1 : wb2);
    const V od = vmul(axis ? w31 : w32, cu);
    f[I] = vfma(om, vsub(vadd(ev, od), f[I]), f[I]);
    f[J] = vfma(om, vsub(vsub(ev, od), f[J]), f[J]);
  });
}

// Shifted-velocity BGK collision of one fluid site, in place on f. a[d] holds the sums
// (a^r, a^b) = sum_i w_i Psi^{r|b}(x + e_i) e_i. A^c = sum_cbar g^{c cbar} a^cbar of
// Eq. (3): the cross coupling g (= g^{rb} = g^{br}) times the other component's sum, plus
// the self coupling g^{cc} times its own.
__device__ __forceinline__ void collide(const LatDev& L, float2 (&f)[Q], float2 rho, float2 ps, const float2 (&a)[3]) {
  float2 m[3], A[3], g;
  float up[3];
  momentum(f, m);
  common_velocity(L, rho, m, up);
  if (L.Gs[0] == 0.0f && L.Gs[1] == 0.0f) {  // the paper's model: the cross coupling alone
    g = make_float2(L.G, L.G);
#pragma unroll
    for (int d = 0; d < 3; ++d) A[d] = make_float2(a[d].y, a[d].x);
  } else {
    g = make_float2(1.0f, 1.0f);
#pragma unroll
    for (int d = 0; d < 3; ++d)
      A[d] = make_float2(__fmaf_rn(L.Gs[0], a[d].x, __fmul_rn(L.G, a[d].y)),
                         __fmaf_rn(L.Gs[1], a[d].y, __fmul_rn(L.G, a[d].x)));
  }
  relax_core(make_float2(L.omega[0], L.omega[1]), make_float2(L.tau[0], L.tau[1]), f, rho, ps, g, A, up);
}

// sum_i w_i Psi^c(x + e_i) e_i of both components (V = float2) or of one (float); psi(I)
// yields Psi of the site x - e_I. Opposite pairs (I, I+1) contribute
// w_I (Psi(x + e_I) - Psi(x - e_I)) e_I.
template <class V, class PsiFrom>
__device__ __forceinline__ void force_sums_by_direction(PsiFrom psi, V (&a)[3]) {
  a[0] = a[1] = a[2] = vset<V>(0.f);
  Unroll<0, 9>::run([&](auto kc) {
    constexpr int I = 1 + 2 * decltype(kc)::value;
    constexpr int ex = dir_x(I), ey = dir_y(I), ez = dir_z(I);
    const V up = psi(std::integral_constant<int, I + 1>());
    const V d = vsub(up, psi(std::integral_constant<int, I>()));
    auto acc = [&](V& v, int e) { v = vfma(vset<V>(e > 0 ? wgt(I) : -wgt(I)), d, v); };
    if (ex != 0) acc(a[0], ex);
    if (ey != 0) acc(a[1], ey);
    if (ez != 0) acc(a[2], ez);
  });
}
// The same from a Psi ring, cells psi(plane slot, ly, lx).
template <class V, class PsiAt>
__device__ __forceinline__ void force_sums(PsiAt psi, int sm1, int s0, int sp1, int ly, int lx, V (&a)[3]) {
  force_sums_by_direction([&](auto ic) {
    constexpr int I = decltype(ic)::value;
    constexpr int ez = dir_z(I);
    return psi(ez > 0 ? sm1 : (ez < 0 ? sp1 : s0), ly - dir_y(I), lx - dir_x(I));
  }, a);
}

// ------------------------------------------------------------------ fused step, one x-y tile column
//
// A CTA of TX*TY threads owns sites [x0, x0+TX) x [y0, y0+TY) and marches z over
// [zb, ze). Psi of the tile plus a one-site halo lives in a 4-plane shared ring,
// so the 18-neighbour force never reads Psi from HBM; halo densities are
// recomputed from the neighbours' pulled populations (an L2 hit when the
// neighbouring CTA is at the same plane). Halo slot h belongs to thread h: the
// two halo rows each fill a warp with contiguous sites, so their pulls coalesce
// like the interior's (spreading them over all warps instead made every halo
// load touch a sector per lane). One barrier per plane: plane z+1 is written
// while plane z-2's slot is free.
//
// The pulls of the next plane are asynchronous copies into shared slots that
// belong to the issuing thread alone (its site's 19 pairs, and its halo
// site's), started as soon as the current plane has been read out of them, so
// their latency overlaps the collision of the previous plane without holding
// registers. Only the thread that issued a copy reads its slot, so a wait on its
// own copies is the only synchronisation the slots need.
template <int TX, int TY, class S>
struct Tile {
  static constexpr int NT = TX * TY, NW = NT / 32, RW = TX + 2, RH = TY + 2, NH = 2 * TX + 2 * RH;
  static constexpr int HS = (NH + 31) / 32 * 32;  // halo slot stride
  static_assert(NH <= NT, "halo slots exceed threads");
  static_assert(NT % 32 == 0, "whole warps");

  struct Smem {
    float2 ring[4][RH][RW];  // (Psi^r, Psi^b) of plane slot, tile row + 1, tile column + 1
    double red[NW];
    typename S::T fin[Q][NT];      // pulled pairs of the own site, [i][thread]
    typename S::T fh[Q][HS];       // pulled pairs of the halo site, [i][thread]
  };

  const LatDev& L;
  Smem& sm;
  const typename S::T* __restrict__ src;
  typename S::T* __restrict__ dst;
  int tx, ty, x, y, hx, hy, hlx, hly;
  bool active, has_halo;
  double evap;

  __device__ __forceinline__ Tile(const LatDev& L_, Smem& sm_, const typename S::T* s_, typename S::T* d_,
                                  const CUtensorMap* = nullptr)
      : L(L_), sm(sm_), src(s_), dst(d_), evap(0.0) {}

  __device__ __forceinline__ int wrapz(int z) const { return z < 0 ? z + L.nz : (z >= L.nz ? z - L.nz : z); }
  __device__ __forceinline__ typename S::T* own_slot() { return &sm.fin[0][threadIdx.x]; }
  __device__ __forceinline__ typename S::T* halo_slot() { return &sm.fh[0][threadIdx.x]; }

  // Bind the CTA to tile column (bx, by). Lanes past a ragged edge stage the
  // wrapped site there (its Psi is the halo of the last real site).
  __device__ __forceinline__ void setup(int bx, int by) {
    const int tid = threadIdx.x;
    tx = tid % TX;
    ty = tid / TX;
    const int gx = bx * TX + tx, gy = by * TY + ty;
    active = gx < L.nx && gy < L.ny;
    x = gx % L.nx;
    y = gy % L.ny;
    // halo slot h = tid: top row, bottom row, left column, right column
    const int h = tid;
    has_halo = h < NH;
    if (h < TX) { hlx = h; hly = -1; }
    else if (h < 2 * TX) { hlx = h - TX; hly = TY; }
    else if (h < 2 * TX + RH) { hlx = -1; hly = h - 2 * TX - 1; }
    else { hlx = TX; hly = h - 2 * TX - RH - 1; }
    hx = wrapi(bx * TX + hlx, L.nx);
    hy = wrapi(by * TY + hly, L.ny);
  }

  // Start the pulls of plane p (p in [-1, nz]) for the own site and the halo site.
  __device__ __forceinline__ void issue(int p, int& cls, int& hcl) {
    const int zp = wrapz(p);
    cls = site_class(L, x, y, zp);
    if (cls != SOLID) pull_async<S>(L, src, PullIdx(L, x, y, zp), own_slot(), NT);
    if (has_halo) {
      hcl = site_class(L, hx, hy, zp);
      if (hcl != SOLID) pull_async<S>(L, src, PullIdx(L, hx, hy, zp), halo_slot(), HS);
    }
    cp_async_commit();
  }

  // Read plane p out of the slots (after the wait): the own site into f, the
  // halo site as sums; apply the sink and publish Psi to ring slot p & 3.
  __device__ __forceinline__ void take(int p, bool own, int cls, int hcl, float2 (&f)[Q], float2& rho) {
    const int slot = p & 3;
    float2 ps = make_float2(0.0f, 0.0f);
    if (cls == SOLID) {
      rho = ps;
    } else {
      const typename S::T* w = own_slot();
#pragma unroll
      for (int i = 0; i < Q; ++i) f[i] = S::cv(w[i * NT], wgt(i));
      rho = sum19(f);
      if (cls == SINK) {
        if (active && own && own_z(L, wrapz(p))) evap += (double)sink_excess(L, f);
        sink_densities(L, rho);
      }
      ps = psi_of(rho);
    }
    sm.ring[slot][ty + 1][tx + 1] = ps;
    if (has_halo) {
      float2 hps = make_float2(0.0f, 0.0f);
      if (hcl != SOLID) {
        const typename S::T* w = halo_slot();
        // the owner's arithmetic, so the halo Psi has the owner's bits
        float2 hrho = sum19_of<float2>([&](auto ic) {
          constexpr int I = decltype(ic)::value;
          return S::cv(w[I * HS], wgt(I));
        });
        if (hcl == SINK) sink_densities(L, hrho);
        hps = psi_of(hrho);
      }
      sm.ring[slot][hly + 1][hlx + 1] = hps;
    }
  }

  // Collide plane z (in [0, nz); read out one plane earlier) and store f*.
  __device__ __forceinline__ void finish(int z, float2 (&f)[Q], float2 rho, int cls) {
    if (!active || cls == SOLID) return;
    const int s = x + L.nx * y + L.nxny * z;
    if (cls == SINK) {
      // Sinks are neither forced nor collided: they stream f^eq(rho_H, 0) and
      // f^eq(rho^r + rho^b - rho_H, 0) as they are.
#pragma unroll
      for (int i = 0; i < Q; ++i) f[i] = rest_pop(i, rho);
    } else {
      float2 a[3];
      auto psi = [&](int sl, int ly, int lx) { return sm.ring[sl][ly + 1][lx + 1]; };
      force_sums(psi, (z - 1) & 3, z & 3, (z + 1) & 3, ty, tx, a);
      collide(L, f, rho, sm.ring[z & 3][ty + 1][tx + 1], a);
    }
    store_site<S>(L, dst, s, f);
  }

  // March planes [zb, ze) upward (down = false) or downward. Plane p is read out
  // of the slots at step o, its successor's pulls are started, and after the
  // barrier plane p - d (whose Psi neighbours are now all in the ring) collides.
  // The halo plane on each end is staged for Psi only. The ring slot of plane
  // p is p & 3 for p = -1 too, as in finish().
  __device__ __forceinline__ bool run(int zb, int ze, bool down) {
    float2 c[Q], n2[Q];
    float2 crho = make_float2(0.f, 0.f), nrho = crho;
    int ccl = SOLID, ncl = SOLID, hcl = SOLID;
    const int d = down ? -1 : 1;
    const int first = down ? ze - 1 : zb;
    const int n = ze - zb;
    issue(first - d, ncl, hcl);
    for (int o = 0; o < n + 2; ++o) {
      const int p = first + (o - 1) * d;
      cp_async_wait_all();
      take(p, o >= 1 && o <= n, ncl, hcl, n2, nrho);
      const int pcl = ncl;
      if (o + 1 < n + 2) issue(p + d, ncl, hcl);
      __syncthreads();
      if (o >= 2) finish(p - d, c, crho, ccl);
#pragma unroll
      for (int i = 0; i < Q; ++i) c[i] = n2[i];
      crho = nrho;
      ccl = pcl;
    }
    return true;
  }

  // Block sum of the evaporated mass (fixed order: warps, then warp 0's lanes).
  __device__ __forceinline__ double block_evap() {
    double v = evap;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sm.red[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
      for (int k = 0; k < NT / 32; ++k) t += sm.red[k];
    return t;
  }
};

// ------------------------------------------------------------------ fused step, staged rows
//
// The same march as Tile, with the pulls staged cooperatively. For each of the 19
// directions the plane's source rows -- the TY + 2 rows y0 - 1 .. y0 + TY shifted by
// -e_y, in plane z - e_z -- are copied into shared memory over columns x0 - E ..
// x0 + TX + E (E pairs are 16 bytes), and the x shift -e_x is applied when a thread
// reads them. The E-column margins hold the side halo, so the halo needs no pulls of its
// own. One direction is one TMA box. Requires nx % E == 0 (then the
// box starts on a 16-byte boundary). A population whose source plane is solid is the
// site's own opposite population (halfway bounce-back): read directly.
//
// TMA fills what lies outside the lattice with zeros, so each thread also fetches its
// share of 16-byte pieces with cp.async into a side buffer -- the left margin of the
// first tile in x, the right margin of every other one, and at the y edges the outermost
// rows, all periodic -- and moves them into the staged rows once the boxes have landed.
// Only the last right margin needs that; the others fetch theirs so that all tiles take
// the same time: with the pieces at lattice edges alone, edge tiles ran 10% slower, fell
// planes behind their neighbours, and the rows and 128-byte lines that neighbours share
// were read from DRAM again (224^3 FP32, 64 x 4 tiles: 2.62 GB read per step against 1.87, of 1.71
// needed, 869 us against 664; with the spherical sink 955 against 714).
//
// Per plane: wait for the copies, read out plane p (Psi to the ring, own populations
// to registers), barrier, start plane p + d's copies, collide plane p - d.
//
// Shift: the step of a lattice in its own storage, shifted by some planes (k_shift). Two
// copied planes past the end of the march stand in for the planes across the periodic seam,
// which the march has overwritten by the time it gets there.
template <int TX, int TY, class S, bool Shift = false>
struct TileRows {
  using T = typename S::T;
  using Index = std::conditional_t<Shift, long long, uint32_t>;  // of a site; copied planes may lie below plane 0
  static constexpr int E = 16 / (int)sizeof(T);           // pairs per 16 bytes
  static constexpr int NT = TX * TY, NW = NT / 32, RW = TX + 2, RH = TY + 2, NH = 2 * TX + 2 * RH;
  static constexpr int SW = TX + 2 * E;                   // staged row width
  static constexpr int CH = SW / E;                       // 16-byte pieces per staged row
  static constexpr int NR = Q * RH;                       // staged rows per plane
  static constexpr int BOX = RH * SW;                     // pairs per box
  static constexpr int IS = (BOX * (int)sizeof(T) + 127) / 128 * 128 / (int)sizeof(T);  // box stride (128-byte aligned)
  static constexpr int YR = 19;                           // wrapped rows per y edge: 5 directions x 2 + 9 x 1
  static_assert(TX % E == 0, "tile width must be a multiple of the chunk");
  static_assert(NH <= NT && NT % 32 == 0, "tile shape");

  struct Smem {
    T stage[Q * IS];         // rows of plane p: [i][y - y0 + 1][x - x0 + E], box i at i IS
    float2 ring[4][RH][RW];  // (Psi^r, Psi^b) of plane slot, tile row + 1, tile column + 1
    double red[NW];
    uint64_t bar;            // completes when a plane's boxes have landed
    alignas(16) T side[1];   // wrapped pieces: x edges [edge][row][E], then y edges [edge][row][SW]
  };
  // Bytes of shared memory for xe sides in x and ye edges in y of one tile (1, or 2 where
  // one tile spans the lattice).
  static constexpr size_t smem_bytes(int xe, int ye) {
    return sizeof(Smem) + sizeof(T) * ((size_t)xe * NR * E + (size_t)ye * YR * SW);
  }

  const LatDev& L;
  Smem& sm;
  const T* src;  // Shift: src and dst overlap
  T* dst;
  const CUtensorMap* map;
  int tx, ty, x, y, hx, hy, hlx, hly, x0, y0;
  int tw, th;                  // the tile's sites in x and y
  bool left, right, low, high; // margins and edge rows that come through the side buffer
  unsigned parity;             // of the plane in flight
  bool active, has_halo, downward;
  double evap;

  __device__ __forceinline__ TileRows(const LatDev& L_, Smem& sm_, const T* s_, T* d_, const CUtensorMap* m_)
      : L(L_), sm(sm_), src(s_), dst(d_), map(m_), parity(0), evap(0.0) {
    if (threadIdx.x == 0) mbar_init(&sm.bar, 1);
    __syncthreads();
  }

  __device__ __forceinline__ int wrapz(int z) const { return z < 0 ? z + L.nz : (z >= L.nz ? z - L.nz : z); }
  // Plane of the source buffer that plane zp - dz is read from (zp: near_plane of the march's).
  __device__ __forceinline__ int near_plane(int p) const { return Shift ? p : wrapz(p); }
  __device__ __forceinline__ int source_plane(int zp, int dz) const {
    const int z = zp - dz;
    if constexpr (Shift) return downward ? (z >= L.nz ? z - L.nz : z) : (z < 0 ? z + L.nz : z);
    return wrapz(z);
  }

  __device__ __forceinline__ void setup(int bx, int by) {
    const int tid = threadIdx.x;
    tx = tid % TX;
    ty = tid / TX;
    const int gx = bx * TX + tx, gy = by * TY + ty;
    active = gx < L.nx && gy < L.ny;
    x = gx % L.nx;
    y = gy % L.ny;
    x0 = bx * TX;
    y0 = by * TY;
    tw = min(TX, L.nx - x0);
    th = min(TY, L.ny - y0);
    left = x0 == 0;
    right = !left || x0 + TX >= L.nx;
    low = y0 < 2;
    high = y0 + TY + 2 > L.ny;
    const int h = tid;  // halo slot: top row, bottom row, left column, right column
    has_halo = h < NH;
    if (h < TX) { hlx = h; hly = -1; }
    else if (h < 2 * TX) { hlx = h - TX; hly = TY; }
    else if (h < 2 * TX + RH) { hlx = -1; hly = h - 2 * TX - 1; }
    else { hlx = TX; hly = h - 2 * TX - RH - 1; }
    hx = wrapi(bx * TX + hlx, L.nx);
    hy = wrapi(by * TY + hly, L.ny);
  }

  // Wrapped rows of a y edge, k in [0, YR): direction i and staged row r. At the low edge the rows of tile rows -1 (e_y >= 0) and 0 (e_y > 0), whose sources
  // lie below row 0; at the high edge those of tile rows th and th - 1.
  __device__ __forceinline__ static void wrapped_row(int k, bool hi_edge, int& i, int& which) {
    // directions with e_y = +1: 3 7 10 15 17, with e_y = -1: 4 8 9 16 18, e_y = 0 the rest
    constexpr unsigned long long up = 3ull | 7ull << 5 | 10ull << 10 | 15ull << 15 | 17ull << 20;
    constexpr unsigned long long dn = 4ull | 8ull << 5 | 9ull << 10 | 16ull << 15 | 18ull << 20;
    constexpr unsigned long long z0 =
        0ull | 1ull << 5 | 2ull << 10 | 5ull << 15 | 6ull << 20 | 11ull << 25 | 12ull << 30 | 13ull << 35 | 14ull << 40;
    if (k < 9) {
      i = (int)(z0 >> (5 * k)) & 31;
      which = 0;
    } else {
      const int j = k - 9;  // 5 directions, outer row first, then the inner one
      i = (int)((hi_edge ? dn : up) >> (5 * (j % 5))) & 31;
      which = j / 5;
    }
  }
  __device__ __forceinline__ T* staged_row(int i, int r) { return sm.stage + i * IS + r * SW; }
  __device__ __forceinline__ const T* source_row(int i, int r, int zp) const {
    const int zs = source_plane(zp, dir_z_rt(i)), ys = wrap_near(y0 - 1 + r - dir_y_rt(i), L.ny);
    return src + ((long long)i * L.np + (long long)zs * L.nxny + (long long)ys * L.nx);
  }
  // This thread's wrapped pieces of plane zp: fetch them into the side buffer, or move
  // them from there into the staged rows.
  template <bool FETCH>
  __device__ __forceinline__ void side_pieces(int zp) {
    T* side = sm.side;
    for (int e = left ? 0 : 1; e < (right ? 2 : 1); ++e) {
      for (int R = threadIdx.x; R < NR; R += NT) {
        const int i = R / RH, r = R - i * RH;
        T* piece = side + R * E;
        if (FETCH) {
          cp_async16(piece, source_row(i, r, zp) + (e == 0 ? L.nx - E : wrap_near(x0 + tw, L.nx)));
        } else {
          *reinterpret_cast<int4*>(staged_row(i, r) + (e == 0 ? 0 : tw + E)) = *reinterpret_cast<const int4*>(piece);
        }
      }
      side += NR * E;
    }
    for (int e = low ? 0 : 1; e < (high ? 2 : 1); ++e) {
      for (int q = threadIdx.x; q < YR * CH; q += NT) {
        const int k = q / CH, j = q - k * CH;
        int i, which;
        wrapped_row(k, e == 1, i, which);
        const int r = e == 0 ? which : th + 1 - which;
        T* piece = side + q * E;
        if (FETCH) {
          cp_async16(piece, source_row(i, r, zp) + wrap_near(x0 - E + j * E, L.nx));
        } else if (r >= 0 && r < RH) {
          *reinterpret_cast<int4*>(staged_row(i, r) + j * E) = *reinterpret_cast<const int4*>(piece);
        }
      }
      if (low && high) side += YR * SW;
    }
  }

  // Start the copies of plane p (p in [-1, nz]). Box i is issued by lane i / NW of warp
  // i % NW, so no warp issues more than a few.
  __device__ __forceinline__ void issue(int p) {
    const int zp = near_plane(p);
    if (threadIdx.x == 0) mbar_expect(&sm.bar, (unsigned)(Q * BOX * (int)sizeof(T)));
    const int i = (int)(threadIdx.x / 32) + NW * (int)(threadIdx.x % 32);
    if (i < Q)
      tma_load4(sm.stage + i * IS, map, x0 - E, y0 - 1 - dir_y_rt(i),
                source_plane(zp, dir_z_rt(i)) + (Shift ? kGhosts : 0), i, &sm.bar);
    side_pieces<true>(zp);
    cp_async_commit();
  }
  // Wait for them; false when they did not land in time.
  __device__ __forceinline__ bool landed(int p) {
    const bool ok = mbar_wait(&sm.bar, parity);
    parity ^= 1u;
    cp_async_wait_all();
    side_pieces<false>(near_plane(p));
    // the next boxes overwrite what these stores wrote
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    __syncthreads();
    return ok;
  }

  // Pair of direction I arriving at tile cell (lx, ly) (ly, lx in [-1, TY] x [-1, TX]):
  // from the staged rows; next to a wall, a pair whose source plane is solid
  // is the site's (index s) own opposite one instead.
  template <int I>
  __device__ __forceinline__ float2 staged(int ly, int lx) const {
    return S::cv(sm.stage[(ly + 1) * SW + lx + E + (I * IS - dir_x(I))], wgt(I));
  }
  template <int I>
  __device__ __forceinline__ float2 pulled(int ly, int lx, bool sol_m, bool sol_p, Index s) const {
    constexpr int ez = dir_z(I);
    if (ez != 0 && (ez > 0 ? sol_m : sol_p)) {
      const T* p = src + (long long)opp(I) * L.np + s;
      if constexpr (Shift) return ldcg<S>(p, wgt(I));  // other CTAs of the launch write this memory later on
      else return ld<S>(p, wgt(I));
    }
    return staged<I>(ly, lx);
  }

  // Read plane p out of the staged rows: the own site into f, the halo site
  // as sums (the owner's arithmetic, so the halo Psi has the owner's bits); apply the
  // sink and publish Psi to ring slot p & 3. Returns the own site's class.
  __device__ __forceinline__ int take(int p, bool own, float2 (&f)[Q], float2& rho) {
    const int zp = wrapz(p), slot = p & 3;
    const bool sol_m = solid_z(L, zp == 0 ? L.nz - 1 : zp - 1), sol_p = solid_z(L, zp == L.nz - 1 ? 0 : zp + 1);
    const int cls = site_class(L, x, y, zp);
    float2 ps = make_float2(0.0f, 0.0f);
    const bool walls = sol_m || sol_p;  // the same for the whole plane
    if (cls == SOLID) {
      rho = ps;
    } else {
      if (!walls) {
        Unroll<0, Q>::run([&](auto ic) {
          constexpr int I = decltype(ic)::value;
          f[I] = staged<I>(ty, tx);
        });
      } else {
        const Index s = (Index)(x + L.nx * y) + (Index)L.nxny * (Index)source_plane(near_plane(p), 0);
        Unroll<0, Q>::run([&](auto ic) {
          constexpr int I = decltype(ic)::value;
          f[I] = pulled<I>(ty, tx, sol_m, sol_p, s);
        });
      }
      rho = sum19(f);
      if (cls == SINK) {
        if (active && own && own_z(L, zp)) evap += (double)sink_excess(L, f);
        sink_densities(L, rho);
      }
      ps = psi_of(rho);
    }
    sm.ring[slot][ty + 1][tx + 1] = ps;
    if (has_halo) {
      const int hcl = site_class(L, hx, hy, zp);
      float2 hps = make_float2(0.0f, 0.0f);
      if (hcl != SOLID) {
        // the owner's arithmetic, so the halo Psi has the owner's bits
        float2 hrho;
        if (!walls) {
          hrho = sum19_of<float2>([&](auto ic) { return staged<decltype(ic)::value>(hly, hlx); });
        } else {
          const Index s = (Index)(hx + L.nx * hy) + (Index)L.nxny * (Index)source_plane(near_plane(p), 0);
          hrho = sum19_of<float2>([&](auto ic) { return pulled<decltype(ic)::value>(hly, hlx, sol_m, sol_p, s); });
        }
        if (hcl == SINK) sink_densities(L, hrho);
        hps = psi_of(hrho);
      }
      sm.ring[slot][hly + 1][hlx + 1] = hps;
    }
    return cls;
  }

  // Collide plane z (in [0, nz); read out one plane earlier) and store f*.
  __device__ __forceinline__ void finish(int z, float2 (&f)[Q], float2 rho, int cls) {
    if (!active || cls == SOLID) return;
    const int s = x + L.nx * y + L.nxny * z;
    if (cls == SINK) {
#pragma unroll
      for (int i = 0; i < Q; ++i) f[i] = rest_pop(i, rho);
    } else {
      float2 a[3];
      auto psi = [&](int sl, int ly, int lx) { return sm.ring[sl][ly + 1][lx + 1]; };
      force_sums(psi, (z - 1) & 3, z & 3, (z + 1) & 3, ty, tx, a);
      collide(L, f, rho, sm.ring[z & 3][ty + 1][tx + 1], a);
    }
    store_site<S>(L, dst, s, f);
  }

  // Returns false when a plane's copies did not land in time (the CTA stops marching).
  __device__ __forceinline__ bool run(int zb, int ze, bool down) {
    float2 c[Q], n2[Q];
    float2 crho = make_float2(0.f, 0.f), nrho = crho;
    int ccl = SOLID;
    const int d = down ? -1 : 1;
    const int first = down ? ze - 1 : zb;
    const int n = ze - zb;
    downward = down;
    issue(first - d);
    for (int o = 0; o < n + 2; ++o) {
      const int p = first + (o - 1) * d;
      const bool ok = landed(p);
      const int pcl = take(p, o >= 1 && o <= n, n2, nrho);
      // ring complete, staged rows read out
      if (__syncthreads_or(!ok)) {
        if (!ok) mbar_wait(&sm.bar, parity ^ 1u);  // no copy may land after the CTA has gone
        return false;
      }
      if (o + 1 < n + 2) issue(p + d);
      if (o >= 2) finish(p - d, c, crho, ccl);
#pragma unroll
      for (int i = 0; i < Q; ++i) c[i] = n2[i];
      crho = nrho;
      ccl = pcl;
    }
    return true;
  }

  __device__ __forceinline__ double block_evap() {
    double v = evap;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sm.red[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
      for (int k = 0; k < NT / 32; ++k) t += sm.red[k];
    return t;
  }
};

// ------------------------------------------------------------------ in-place (AA) step
//
// One population lattice A updated in place. Between steps A holds, for every
// non-solid site x and direction i, the population arriving at x in direction i
// (the post-collision value of x - e_i, or x's own opposite one next to a wall):
//   even form: at (i, x - e_i), or at (opp(i), x) where x - e_i is solid -- the
//              slots the two-lattice pull reads (PullIdx::at);
//   odd form:  at (opp(i), x).
// A step reads the arrived populations of x and writes its post-collision f*_j
// into the slot that population opp(j) came from. In the even form that slot is
// where f*_j arrives in the odd form (x + e_j, or (j, x) when x + e_j is solid);
// in the odd form it is (j, x), the even form's slot of f*_j. The slots a site
// reads are exactly those it writes and belong to no other site, so no site's
// update touches another's data. Only the force couples sites: every neighbour's
// Psi must be formed before that neighbour is overwritten, so Psi comes from a
// separate pass (k_aa_psi) into an (Psi^r, Psi^b) array.

// Slot of the population arriving at the site of P in direction I.
template <int I, bool ODD>
__device__ __forceinline__ void aa_slot(const PullIdx& P, int& idx, int& d) {
  if (ODD) {
    idx = P.s;
    d = opp(I);
  } else {
    P.template at<I>(idx, d);
  }
}

// Arrived populations of the site of P (plain loads: the lattice is written in place).
template <class S, bool ODD>
__device__ __forceinline__ void aa_load(const LatDev& L, const typename S::T* A, const PullIdx& P,
                                        float2 (&f)[Q]) {
  Unroll<0, Q>::run([&](auto ic) {
    constexpr int I = decltype(ic)::value;
    int idx, d;
    aa_slot<I, ODD>(P, idx, d);
    f[I] = S::cv(A[(long long)d * L.np + idx], wgt(I));
  });
}

// The same loads at L2 only (the persistent in-place step, where neighbouring CTAs
// rewrite slots this CTA read in an earlier step).
template <class S, bool ODD>
__device__ __forceinline__ void aa_load_cg(const LatDev& L, const typename S::T* A, const PullIdx& P,
                                           float2 (&f)[Q]) {
  Unroll<0, Q>::run([&](auto ic) {
    constexpr int I = decltype(ic)::value;
    int idx, d;
    aa_slot<I, ODD>(P, idx, d);
    f[I] = ldcg<S>(A + (long long)d * L.np + idx, wgt(I));
  });
}

// f*_j into the slot population opp(j) was read from.
template <class S, bool ODD>
__device__ __forceinline__ void aa_store(const LatDev& L, typename S::T* A, const PullIdx& P,
                                         const float2 (&f)[Q]) {
  Unroll<0, Q>::run([&](auto jc) {
    constexpr int J = decltype(jc)::value;
    int idx, d;
    aa_slot<opp(J), ODD>(P, idx, d);
    put<S>(A + (long long)d * L.np + idx, f[J], wgt(J));
  });
}

}  // namespace sclbm
