// Resident step of small lattices: one launch advances many steps with the populations
// held in the shared memory of one thread-block cluster. Included by sc_lbm.cu, whose
// handle and helpers it shares.
//
// A lattice of a few thousand sites is bound by latency: a launch per step cost 10.5 us
// (4x4x128, FP32, graphs of 64 launches), of which the arithmetic is under 1 us. Here CTA
// r of a cluster of C holds sites [r ML, (r + 1) ML), one per thread, as two buffers
// f[direction][site] of pairs in the storage type plus Psi; a step is
//   pull the 19 directions of both components from the current buffer (the own CTA's or
//   another's shared memory), densities, sink, Psi | cluster barrier | force from the
//   neighbours' Psi, collision, store to the other buffer | cluster barrier.
// Where a CTA holds whole planes and has threads to spare for the plane on each side (PLANES),
// these form that plane's Psi from its populations (the owner's arithmetic, so its bits): Psi
// is then shared within the CTA and the first cluster barrier is a CTA barrier: 100 film steps
// with diagnostics and read-out 168 -> 155 us.
// The addresses of the 19 sources are the same in every step and stay in registers (a
// population next to a wall is the site's own opposite one, and a solid neighbour's Psi a
// cell that holds 0), so a step has no index arithmetic. Values are rounded to the
// storage type when stored and the arithmetic is the other kernels', so the bits are theirs.

namespace {

constexpr int kResidentThreads = 512;   // most sites per CTA
constexpr int kResidentCluster = 16;    // most CTAs (non-portable size)
constexpr int kResidentMaxSteps = 4096; // steps per launch

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned map_rank(unsigned addr, unsigned rank) {
  unsigned r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
__device__ __forceinline__ float2 ld_cluster(unsigned addr, float2) {
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t ld_cluster(unsigned addr, uint32_t) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}

// Bytes of shared memory for ML sites: the two buffers, then (Psi^r, Psi^b) of ML sites
// and of `extra`: the planes on each side, or the cell that holds 0.
__host__ __device__ constexpr size_t resident_pop_bytes(int es, int ML) {
  return ((size_t)2 * 2 * Q * ML * es + 15) / 16 * 16;
}
constexpr size_t resident_smem(int es, int ML, int extra) {
  return resident_pop_bytes(es, ML) + sizeof(float2) * ((size_t)ML + extra);
}

template <class S, bool PLANES>
__global__ void __launch_bounds__(kResidentThreads, 1)
    k_resident(const LatDev L, typename S::T* __restrict__ pop, double* __restrict__ evap_cum, int K, int ML) {
  using T = typename S::T;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  T* f_sm = reinterpret_cast<T*>(smem_raw);
  float2* psi_sm = reinterpret_cast<float2*>(smem_raw + resident_pop_bytes((int)sizeof(T) / 2, ML));
  const int n = L.nxny * L.nz, local = (int)threadIdx.x;
  const unsigned rank = cluster_rank();
  const int s = (int)rank * ML + local;
  const bool held = local < ML && s < n;
  int x = 0, y = 0, z = 0;
  if (held) site_of(L, s, x, y, z);
  // Psi cell: own sites in order, with PLANES after the plane below, and the one above next
  const int mine = min(ML, n - (int)rank * ML);  // the CTA's sites (whole planes with PLANES)
  int cell = PLANES ? local + L.nxny : local;
  bool halo = false;
  if (PLANES && local >= ML && mine > 0) {
    const int q = local - ML;  // a site of the plane below or above
    halo = q < 2 * L.nxny;
    if (halo) {
      const bool above = q >= L.nxny;
      const int in_plane = above ? q - L.nxny : q;
      const int zb = ((int)rank * ML) / L.nxny, ze = zb + mine / L.nxny;
      x = in_plane % L.nx;
      y = in_plane / L.nx;
      z = above ? (ze == L.nz ? 0 : ze) : (zb == 0 ? L.nz - 1 : zb - 1);
      cell = in_plane + (above ? L.nxny + mine : 0);
    }
  }
  const int cls = held || halo ? site_class(L, x, y, z) : SOLID;
  const bool live = cls != SOLID;

  unsigned fa[Q], pa[Q];  // source pair (buffer 0) and Psi of site x - e_I
  const unsigned f_base = smem_addr(f_sm), p_base = smem_addr(psi_sm);
  {
    const PullIdx P(L, x, y, z);
    Unroll<0, Q>::run([&](auto ic) {
      constexpr int I = decltype(ic)::value;
      int idx, d;
      P.template at<I>(idx, d);
      const int owner = idx / ML, loc = idx - owner * ML;
      fa[I] = map_rank(f_base + (unsigned)((d * ML + loc) * (int)sizeof(T)), (unsigned)owner);
      if constexpr (PLANES) {  // site x - e_I within the CTA; 0 is stored at solid sites
        const int xs = P.xs[1 + dir_x(I)], ys = P.ys[1 + dir_y(I)];
        pa[I] = p_base + (unsigned)((held ? cell - y * L.nx - x - dir_z(I) * L.nxny + ys + xs : 0) * (int)sizeof(float2));
      } else
      pa[I] = d == I ? map_rank(p_base + (unsigned)(loc * (int)sizeof(float2)), (unsigned)owner)
                     : p_base + (unsigned)(ML * (int)sizeof(float2));
    });
  }
  if (held) {
#pragma unroll 1
    for (int d = 0; d < Q; ++d) f_sm[d * ML + local] = pop[(long long)d * L.np + s];
  }
  if (!PLANES && threadIdx.x == 0) psi_sm[ML] = make_float2(0.f, 0.f);
  const unsigned bytes = (unsigned)(Q * ML * (int)sizeof(T));
  double evap = 0.0;
  cluster_barrier();
#pragma unroll 1
  for (int k = 0; k < K; ++k) {
    const unsigned boff = (k & 1) ? bytes : 0u;
    float2 f[Q], rho = make_float2(0.f, 0.f), ps = rho;
    if (live) {
      Unroll<0, Q>::run([&](auto ic) {
        constexpr int I = decltype(ic)::value;
        f[I] = S::cv(ld_cluster(fa[I] + boff, T()), wgt(I));
      });
      rho = sum19(f);
      if (cls == SINK) {
        if (held) evap += (double)sink_excess(L, f);
        sink_densities(L, rho);
      }
      ps = psi_of(rho);
    }
    if (held || halo) psi_sm[cell] = ps;
    if constexpr (PLANES) __syncthreads();
    else cluster_barrier();
    if (live && held) {
      if (cls == SINK) {
#pragma unroll
        for (int i = 0; i < Q; ++i) f[i] = rest_pop(i, rho);
      } else {
        float2 a[3];
        force_sums_by_direction([&](auto ic) {
          constexpr int I = decltype(ic)::value;
          return ld_cluster(pa[I], float2());
        }, a);
        collide(L, f, rho, ps, a);
      }
      T* to = f_sm + ((k & 1) ? 0 : Q * ML) + local;
#pragma unroll
      for (int i = 0; i < Q; ++i) to[i * ML] = S::enc(f[i], wgt(i));
    }
    cluster_barrier();
  }
  if (held) {
    const T* from = f_sm + ((K & 1) ? Q * ML : 0) + local;
#pragma unroll 1
    for (int d = 0; d < Q; ++d) pop[(long long)d * L.np + s] = from[d * ML];
  }
  if (L.geometry != 0) {
    __shared__ double red[kResidentThreads / 32];
    double v = evap;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int w = 0; w < (int)blockDim.x / 32; ++w) t += red[w];
      evap_cum[rank] += t;
    }
  }
}

template <bool PLANES>
void* resident_fn_of(int storage) {
  switch (storage) {
    case SC_STORAGE_F16: return (void*)k_resident<StF16, PLANES>;
    case SC_STORAGE_F16_SCALED: return (void*)k_resident<StF16S, PLANES>;
    case SC_STORAGE_BF16: return (void*)k_resident<StBF16, PLANES>;
    default: return (void*)k_resident<StF32, PLANES>;
  }
}
void* resident_fn(const sc_lbm* h) {
  return h->rplanes ? resident_fn_of<true>(h->p.storage) : resident_fn_of<false>(h->p.storage);
}

void resident_config(const sc_lbm* h, cudaLaunchConfig_t* cfg, cudaLaunchAttribute* at, cudaStream_t st) {
  *cfg = cudaLaunchConfig_t{};
  cfg->gridDim = dim3((unsigned)h->rcta);
  const int extra = 2 * h->L.nxny;
  cfg->blockDim = dim3((unsigned)round_up(h->rsites + (h->rplanes ? extra : 0), 32));
  cfg->dynamicSmemBytes = resident_smem((int)elem_size(h->p.storage), h->rsites, h->rplanes ? extra : 1);
  cfg->stream = st;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = (unsigned)h->rcta;
  at->val.clusterDim.y = at->val.clusterDim.z = 1;
  cfg->attrs = at;
  cfg->numAttrs = 1;
}

// Plans the resident step of a two-lattice handle: a cluster of up to 16 CTAs, 128 sites
// per CTA while that suffices (one warp per scheduler), up to 512. Leaves h->rcta = 0 where
// the lattice is too large, the caller chose a kernel (staging, tile or planes per CTA) or the
// device cannot hold the cluster.
void plan_resident(sc_lbm* h) {
  h->rcta = 0;
  const sc_params& p = h->p;
  if (h->lay.aa || p.staging != SC_STAGING_AUTO || p.tile != 0 || p.zchunk != 0) return;
  const long long n = h->lay.nsites;
  if (n > (long long)kResidentCluster * kResidentThreads) return;
  int c = 1;
  while (c < kResidentCluster && n > 128LL * c) c *= 2;
  for (; c >= 1; c /= 2) {
    const long long ml = (n + c - 1) / c, plane = h->L.nxny, whole = (ml + plane - 1) / plane * plane;
    if (ml > kResidentThreads || c > h->lay.nslots) continue;
    h->rcta = c;
    h->rplanes = whole + 2 * plane <= kResidentThreads;
    h->rsites = (int)(h->rplanes ? whole : ml);
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at;
    resident_config(h, &cfg, &at, h->stream);
    void* fn = resident_fn(h);
    const int most = (int)resident_smem((int)elem_size(p.storage), kResidentThreads, 1);
    int clusters = 0;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, most) == cudaSuccess &&
        cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&clusters, fn, &cfg) == cudaSuccess && clusters >= 1)
      return;
    cudaGetLastError();
    h->rcta = 0;
  }
}

// Whether a call of nsteps steps takes the resident launch. A single step is not worth the way into
// shared memory and back (us for one step, resident / two-lattice: 20^3 FP32 16.7 / 8.5, 4x4x128 10.5 /
// 8.5; for two steps 20.8 / 16.8 and 12.1 / 16.7), unless the two-lattice tiles of 8 x 4 sites are
// nearly empty and many (1x1x100 16.6 / 15.9, 1x1x1000 18.3 / 26.5, 1x1x8000 19.9 / 67.7, 1x8x1000
// 19.7 / 25.7, 1x64x100 18.8 / 22.6, 2x2x2000 20.0 / 21.2; against 8x1x1000 19.8 / 17.0, 2x3x1300
// 19.9 / 18.1; with the host's wait, 6 us).
bool resident_takes(const sc_lbm* h, int64_t nsteps) {
  if (h->rcta == 0 || nsteps != 1) return h->rcta > 0;
  const long long lanes = 32LL * ((h->p.nx + 7) / 8) * ((h->p.ny + 3) / 4) * h->p.nz;
  return lanes >= 16000 && lanes >= 8 * h->lay.nsites;
}

// nsteps steps in place on the current buffer.
int launch_resident(sc_lbm* h, int64_t nsteps) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at;
  resident_config(h, &cfg, &at, h->stream);
  for (int64_t left = nsteps; left > 0; left -= kResidentMaxSteps) {
    LatDev L = h->L;
    void* pop = h->pop(h->cur);
    double* evap = h->evap();
    int K = (int)std::min<int64_t>(left, kResidentMaxSteps), ML = h->rsites;
    void* args[] = {&L, &pop, &evap, &K, &ML};
    const cudaError_t e = cudaLaunchKernelExC(&cfg, resident_fn(h), args);
    if (e != cudaSuccess) return fail(SC_ECUDA, "resident step launch failed: %s", cudaGetErrorString(e));
  }
  return SC_OK;
}

}  // namespace
