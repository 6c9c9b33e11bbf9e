// Shifted step: one population lattice advanced in its own storage by the two-lattice step's
// staged-rows march. Included by sc_lbm.cu, whose handle and helpers it shares.
//
// The 19 arrays of pairs have nz + s + 4 planes. In state 0 the lattice lies in planes [2, nz + 2), in
// state 1 in planes [s + 2, nz + s + 2); a step reads one and writes the other, so plane z is
// written s planes away from where it is read, over old plane z - s (state 1 -> 0, marching up)
// or z + s (0 -> 1, marching down). The work is cut into chunks of at most s - 2 planes, claimed
// in march order: the old planes that an item of chunk k overwrites lie before those that chunk
// k and later ones read (their planes and two more on each side). So an item waits until the
// items of the tile columns within two of its own, which alone read its sites, have finished
// the chunk before (and with that, by the same rule, all earlier ones). Items wait only on
// items claimed before them, by CTAs that are running, so the waits end; each is still bounded.
// The march's last chunk needs old planes from across the periodic seam that its first chunk
// overwrote: k_shift_begin copies those two planes past the end before the step.
//
// Why: in place, the force needs Psi of a neighbour before that neighbour is overwritten, so
// the AA steps read every population twice, and on a 512^2 plane (40 MB per plane, three in
// use) the second read misses the L2. Here it is read once, plus the halo planes of the chunks:
// 512^3 FP32, 20 steps 234 (persistent) -> 180 ms, 9.0 ms per step against a floor of 6.0 and the
// two-lattice step's 6.9 (a slower GPU of the kind took 215). Beyond that it reads more: 512 x 288 x 201
// FP16, chunks of up to 15 planes, 3.3 to 3.4 GB per step for 2.25 needed, 1.28 times of it the
// planes on each side of a chunk, the rest rows that neighbouring tiles no longer find in the
// L2; it writes 2.27 GB. The march spills 94 bytes a thread (FP32 and scaled FP16; 90 FP16 and BF16).

namespace {

// Longest chunk: shorter ones read too many halo planes ((c + 4) / c; FP32 320^3, 10 planes: 3.36
// against 2.85 ms for the two-pass step, 384^3, 12: 4.54 against 4.33; 448^3, 16: 6.2 against 7.6).
constexpr int kShiftMinChunk = 15;
// Tile columns: about two rounds of the resident CTAs (2 on each of 152 SMs), so that the chunk
// before is finished around an item's column when the item is claimed. With fewer the items
// wait for one another (FP16 320^3, 400 columns: 2.31 against 2.31 ms for the two-pass step;
// 384^3, 576: 3.16 against 3.41; 512 x 512 x 256, 1024: 3.35 against 4.03).
constexpr int kShiftMinCols = 576;
constexpr int kShiftReach = 2;     // tile columns on each side whose items may read a tile's sites

// Planes that the lattice moves by: the Psi array's memory as extra planes of the 19 arrays,
// less the copied ones. 0 where the shifted step does not apply.
int shift_planes(const sc_params* p, long long es, long long bytes, long long* np) {
  if (p->layout != SC_LAYOUT_AA || p->staging != SC_STAGING_AUTO || p->tile != 0 || p->zchunk != 0 || p->nx < 64 ||
      p->nx % (8 / es) != 0)
    return 0;
  const long long cols = (long long)((p->nx + 63) / 64) * ((p->ny + 3) / 4);
  if (cols > 2 * kMaxCtas || cols < kShiftMinCols) return 0;
  const long long room = bytes / (2 * Q * es) / (128 / es) * (128 / es);
  const long long s = std::min<long long>(room / ((long long)p->nx * p->ny) - p->nz - 2 * kGhosts, p->nz);
  if (s < kShiftMinChunk + 2) return 0;
  *np = room;
  return (int)s;
}

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_u32(unsigned* p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

struct ShiftArgs {
  int cols_x, cols_y, nch;
  bool down;
  unsigned* next;       // claim counter, 0 between launches
  unsigned* done;       // chunks finished, per tile column
  int* err;             // set to 3 when a plane's copies, to 4 when a neighbour's chunk did not come in time
  long long limit_ns;   // of a wait
  int withhold;         // CTA that reports no finished chunk (-1: none)
};

// Copies `n16` 16-byte pieces (two planes) of each of the Q arrays and clears the column counters.
__global__ void __launch_bounds__(256) k_shift_begin(const int4* __restrict__ from, int4* __restrict__ to,
                                                     long long stride16, int n16, unsigned* __restrict__ done, int cols) {
  const long long t = blockIdx.x * 256LL + threadIdx.x, step = gridDim.x * 256LL;
  for (long long k = t; k < cols; k += step) done[k] = 0u;
  for (long long k = t; k < (long long)Q * n16; k += step) {
    const long long a = k / n16, o = a * stride16 + (k - a * n16);
    to[o] = from[o];
  }
}

template <int TX, int TY, class S>
__global__ void __launch_bounds__(TX * TY, 512 / (TX * TY))
    k_shift(const LatDev L, const typename S::T* src, typename S::T* dst, double* __restrict__ evap_cum,
            const __grid_constant__ ShiftArgs a, const __grid_constant__ CUtensorMap map) {
  using TileT = TileRows<TX, TY, S, true>;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  auto& sm = *reinterpret_cast<typename TileT::Smem*>(smem_raw);
  __shared__ int s_it[2];
  TileT t(L, sm, src, dst, &map);
  const int cols = a.cols_x * a.cols_y, nitems = cols * a.nch;
  // one claim per item and a failing one per CTA; the last wraps the counter to 0
  const unsigned last = (unsigned)nitems + gridDim.x - 1u;
  if (threadIdx.x == 0) s_it[0] = (int)atomicInc(a.next, last);
  __syncthreads();
  int turn = 0;
  bool ok = true;
  for (int it = s_it[0]; it < nitems; it = s_it[turn ^= 1]) {
    if (threadIdx.x == 0) s_it[turn ^ 1] = (int)atomicInc(a.next, last);  // one item ahead
    const int k = it / cols, col = it - k * cols, by = col / a.cols_x, bx = col - by * a.cols_x;
    constexpr int R = 2 * kShiftReach + 1;
    bool got = true;
    if (ok && k > 0 && threadIdx.x < R * R) {
      const int dx = (int)threadIdx.x % R - kShiftReach, dy = (int)threadIdx.x / R - kShiftReach;
      const unsigned* d = a.done + (wrapi(bx + dx, a.cols_x) + a.cols_x * wrapi(by + dy, a.cols_y));
      if (ld_acquire_u32(d) < (unsigned)k) {
        const unsigned long long t0 = global_ns();
        while (got && ld_acquire_u32(d) < (unsigned)k) got = (long long)(global_ns() - t0) <= a.limit_ns;
      }
    }
    if (__syncthreads_or(!got)) {
      ok = false;
      if (threadIdx.x == 0) *a.err = 4;
    }
    if (ok) {
      t.setup(bx, by);
      const int c = a.down ? a.nch - 1 - k : k;
      ok = t.run((int)((long long)c * L.nz / a.nch), (int)((long long)(c + 1) * L.nz / a.nch), a.down);
      if (!ok && threadIdx.x == 0) *a.err = 3;
    }
    if (L.geometry != 0 && __syncthreads_or(t.evap != 0.0)) {
      const double e = t.block_evap();
      if (threadIdx.x == 0) atomicAdd(evap_cum + col, e);  // the column's chunks follow one another
      t.evap = 0.0;
    }
    __syncthreads();  // the item's last reads and stores, and the next item's number
    if (ok && threadIdx.x == 0 && (int)blockIdx.x != a.withhold) st_release_u32(a.done + col, (unsigned)k + 1u);
  }
}

constexpr int kShiftTile = 4;  // kTileX x kTileY = 64 x 4
template <class S>
constexpr size_t shift_smem(const LatDev& L) {
  return TileRows<64, 4, S, true>::smem_bytes(L.nx <= 64 ? 2 : 1, L.ny < 6 ? 2 : 1);
}
template <class S>
int shift_occupancy(const LatDev& L) {
  int nb = 0;
  constexpr size_t most = TileRows<64, 4, S, true>::smem_bytes(2, 2);
  if (cudaFuncSetAttribute(k_shift<64, 4, S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_shift<64, 4, S>, 256, shift_smem<S>(L)) != cudaSuccess)
    return 0;
  return nb;
}

// Chunks: the fewest rounds of the resident CTAs times the planes each item stages, at most
// s - 2 planes each.
int plan_shift(sc_lbm* h) {
  int dev = 0, sms = 1, occ = 0;
  CK(cudaGetDevice(&dev));
  CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  switch (h->p.storage) {
    case SC_STORAGE_F16: occ = shift_occupancy<StF16>(h->L); break;
    case SC_STORAGE_F16_SCALED: occ = shift_occupancy<StF16S>(h->L); break;
    case SC_STORAGE_BF16: occ = shift_occupancy<StBF16>(h->L); break;
    default: occ = shift_occupancy<StF32>(h->L);
  }
  if (occ < 1) return fail(SC_ECUDA, "the shifted step kernel cannot be made resident: %s", cudaGetErrorString(cudaGetLastError()));
  Layout& l = h->lay;
  l.tile = kShiftTile;
  l.tx = kTileX[kShiftTile];
  l.ty = kTileY[kShiftTile];
  l.cols_x = (h->p.nx + l.tx - 1) / l.tx;
  l.cols = l.cols_x * ((h->p.ny + l.ty - 1) / l.ty);
  const long long slots = (long long)sms * occ, nz = h->p.nz, most = l.planes - 2;
  double best = 1e300;
  long long nch = 0;
  for (long long n = (nz + most - 1) / most; n <= nz; ++n) {
    const double cost = (double)((l.cols * n + slots - 1) / slots) * ((double)((nz + n - 1) / n) + 2.0);
    if (cost < best * (1.0 - 1e-9)) { best = cost; nch = n; }
  }
  h->nitems = (int)nch;
  h->zmax = (int)((nz + nch - 1) / nch);
  h->grid = (int)std::min<long long>(slots, l.cols * nch);
  h->wait_limit_ns = 2000000000LL;
  h->withhold = -1;
  for (int k = 0; k < 2; ++k) {
    const int rc = encode_map(h, (char*)h->pop(k) - (size_t)kGhosts * h->L.nxny * 2 * elem_size(h->p.storage), l.tile,
                              &h->maps[k]);
    if (rc) return rc;
  }
  return SC_OK;
}

template <class S>
cudaError_t launch_shift(sc_lbm* h, cudaStream_t st) {
  using T = typename S::T;
  const Layout& l = h->lay;
  const bool down = h->cur == 0;
  const T* src = (const T*)h->pop(h->cur);
  const long long plane = h->L.nxny, nz = h->p.nz;
  constexpr int E = 16 / (int)sizeof(T);
  const T* from = down ? src + (nz - kGhosts) * plane : src;
  T* to = const_cast<T*>(down ? src - kGhosts * plane : src + nz * plane);
  const int n16 = (int)(kGhosts * plane / E);
  unsigned* done = (unsigned*)h->flags();
  k_shift_begin<<<grid_for((long long)Q * n16, 1024), 256, 0, st>>>((const int4*)from, (int4*)to, h->L.np / E, n16, done, l.cols);
  const ShiftArgs a{l.cols_x, l.cols / l.cols_x, h->nitems, down, h->next(), done, h->h_err, h->wait_limit_ns, h->withhold};
  k_shift<64, 4, S><<<h->grid, 256, shift_smem<S>(h->L), st>>>(h->L, src, (T*)h->pop(1 - h->cur), h->evap(), a,
                                                               h->maps[h->cur]);
  return cudaGetLastError();
}

int launch_shift_one(sc_lbm* h, cudaStream_t st) {
  cudaError_t e;
  switch (h->p.storage) {
    case SC_STORAGE_F16: e = launch_shift<StF16>(h, st); break;
    case SC_STORAGE_F16_SCALED: e = launch_shift<StF16S>(h, st); break;
    case SC_STORAGE_BF16: e = launch_shift<StBF16>(h, st); break;
    default: e = launch_shift<StF32>(h, st);
  }
  if (e != cudaSuccess) return fail(SC_ECUDA, "shifted step launch failed: %s", cudaGetErrorString(e));
  h->cur = 1 - h->cur;
  return SC_OK;
}

// The persistent step takes over the lattice where it stands (its even form is the pull's):
// sc_lbm_persist_bands asks for bands, which only that step has. Its saved columns use the
// read-out area.
int shift_to_persist(sc_lbm* h) {
  CK(cudaMemsetAsync(h->flags(), 0, (size_t)2 * kMaxCtas * sizeof(unsigned long long), h->stream));
  Layout& l = h->lay;
  l.off_pop[0] = l.off_pop[1] = l.off_pop[h->cur];
  l.off_psi = l.off_stage;
  l.shift = l.rows = false;
  l.aa = true;
  h->cur = 0;
  if (h->graph) { cudaGraphExecDestroy(h->graph); h->graph = nullptr; }
  return SC_OK;
}

}  // namespace
