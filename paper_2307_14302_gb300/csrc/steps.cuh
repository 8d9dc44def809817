// steps.cuh -- whole steps of a small mesh in one launch of one thread-block cluster.
//
// A mesh of at most a few hundred 32-element tiles does not fill the GPU, and a launch per stage then
// costs more than the stage: on 960 triangles (30 tiles) a stage took 4.6 us of which the arithmetic
// of one tile is under 2.  Here the tiles live in the shared memory of one cluster (at most 16 CTAs,
// one warp per tile) for as many steps as a call asks for: geometry, plan and the stage buffers are
// loaded once, each warp advances its tile with the same tile_body as tile_kernel (so results agree
// bit for bit), out-of-tile neighbours are read from the other CTAs' shared memory, and the stages
// are separated by the cluster's hardware barrier.  A cluster's CTAs are scheduled together, so the
// barrier needs no co-residency argument and no polling.
//
// The barrier is split: a warp arrives when its new record is written and waits only when it needs
// another tile's (after the area integrals and the in-tile edges of the next stage), so the barrier's
// latency and the spread between warps are mostly hidden.  What is written after that wait (the
// record of stage k + 1) may replace what other tiles read before their arrival (stage k's input), so
// two record buffers are enough for a two-stage scheme and three for longer ones.
#pragma once
#include "tile.cuh"

namespace dg {

template <int P, class Pol, int FT = FT_ALL>
struct StepsLayout {
  using L = TileLayout<P, Pol, FT>;
  static constexpr int RECS = TILE * L::RV;                       // one record buffer of a tile, 16-byte units
  static constexpr int GEO = L::S_GEO, PLAN = L::S_PLAN, XY = L::S_XY;
  static constexpr int HAL = L::SV;
  static constexpr int FLX = HAL + HALO * L::RV;
  static constexpr int REC = FLX + (L::BAR - L::FLX);             // 2 or 3 record buffers
  DG_HD static constexpr int vec(int nrec) { return REC + nrec * RECS; }
};
template <int P, class Pol, int FT = FT_ALL>
constexpr int steps_smem_per_warp(int nrec) {
  return 16 * StepsLayout<P, Pol, FT>::vec(nrec);
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// address of the same shared-memory location in CTA `rank` of the cluster, and a 16-byte load from it
__device__ __forceinline__ uint32_t cluster_map(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ uint4 ld_cluster128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}

// register budget: 16 warps per CTA in the mixed p = 1 path, 10 at p = 2, 9 in FP64
template <int P, int FLUX, class Pol, int FT>
__global__ void __maxnreg__(sizeof(typename Pol::T) == 4 ? (P == 1 ? 128 : 200) : 224)
    steps_kernel(const StageArgs<Pol> a0, const StepsArgs st) {
  using T = typename Pol::T;
  using Acc = typename Pol::Acc;
  using L = TileLayout<P, Pol, FT>;
  using SL = StepsLayout<P, Pol, FT>;
  constexpr int NP = np_of(P), NG = P + 1, RV = L::RV;
  const RefTab<T>& tab = ctab<T, P>();
  __shared__ T s_ephi[3][NG][NP];
  __shared__ float4 s_ephi4[P == 1 ? 3 : 15];
  extern __shared__ uint4 tsm[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid; sizeof(T) == 8 && i < 3 * NG * NP; i += blockDim.x) {
    const int j = i / (NG * NP), k = (i / NP) % NG, m = i % NP;
    s_ephi[j][k][m] = tab.ephi[j][k][m];
  }
  edge_rows<P>(tab, s_ephi4);
  const int wpc = blockDim.x >> 5;
  const int tile = blockIdx.x * wpc + warp;  // one tile per warp
  const int vec = SL::vec(st.nrec);
  uint4* Wm = tsm + (size_t)warp * vec;
  uint4* halo = Wm + SL::HAL;
  StageArgs<Pol> a = a0;
  int4 meta = make_int4(0, 0, 0, 0);
  if (tile < a.ntiles) {
    const uint4* from = a.stat + (size_t)tile * L::SVM;
    meta = reinterpret_cast<const int4*>(from)[L::S_META];
    for (int i = lane; i < L::SV; i += 32) Wm[i] = __ldg(from + i);
    for (int i = lane; i < SL::RECS; i += 32) Wm[SL::REC + i] = a.wn[(size_t)tile * SL::RECS + i];
  }
  const int sc = meta.x, present = meta.y, nhalo = meta.z >> 16;
  const bool valid = lane < present;
  __syncthreads();  // edge basis table; the tile's data is read by its own warp and, after the cluster barrier, by others
  cluster_arrive();
  // address, in buffer 0 of its CTA, of the record at a place of the record array, and that of this
  // lane's halo neighbour
  auto remote = [&](uint32_t at) {
    const uint32_t nt = at / (uint32_t)(TILE * RV);
    return cluster_map(smem_u32(tsm + (size_t)(nt % wpc) * vec + SL::REC) + 16u * (at & 31), nt / (uint32_t)wpc);
  };
  const uint32_t hsrc =
      lane < nhalo ? remote(reinterpret_cast<const uint32_t*>(Wm + L::S_HALO)[lane]) : 0u;
  const ScenDev& S = a.scen[sc];
  const unsigned long long step0 = a.ctl->step;
  const int rain_kind = ft_rain(FT) >= 0 ? ft_rain(FT) : S.rain_kind;
  const int press = (FT & FT_PRESS) ? S.press : 0;
  // ledger: a lane's volumes of the launch in three floats (mixed).  A pair over the whole launch rounds a
  // steady rain's equal addends the same way every time, 2e-12 of the volume after 1,000 steps of
  // SSP(5,2), where the tile form, which books in FP64 after every stage, keeps 1e-14.  us per step with a
  // pair and so: 400 triangles 5.0 and 4.9, flume 6.5 and 6.3, 4.8k river LLF SSP(5,2) 21.6 and 22.0 (445
  // and 460 us per 20 steps); an FP64 sum per step took the flume to 6.9, three floats per step instead of
  // per stage the 400 triangles to 5.45.
  typename LongSum<Acc>::type rain_sum = {}, bdry_sum = {};
  for (int n = 0; n < st.nsteps; ++n) {
    for (int s = 0; s < st.nstage; ++s) {
      const StepsArgs::Stage& c = st.st[s];
      const uint32_t rin = 16u * SL::RECS * c.in;
      // the one wait of a stage: every record of the previous one is then written
      auto halo_ready = [&] {
        __syncwarp();
        cluster_wait();
        if (lane < nhalo) {
          uint4 v[RV];
#pragma unroll
          for (int i = 0; i < RV; ++i) v[i] = ld_cluster128(hsrc + rin + 16u * TILE * i);
#pragma unroll
          for (int i = 0; i < RV; ++i) halo[i * HALO + lane] = v[i];
        }
        __syncwarp();
      };
      if (present == 0) {  // no tile, or padding: keep the barrier's count
        __syncwarp();
        cluster_wait();
        cluster_arrive();
        continue;
      }
      a.stage = s;
      a.has_n = c.has_n;
      a.pow2 = c.pow2;
      a.a_n_hi = c.a_n_hi;
      a.a_n_lo = c.a_n_lo;
      a.a_in_hi = c.a_in_hi;
      a.a_in_lo = c.a_in_lo;
      a.a_n = c.a_n;
      a.a_in = c.a_in;
      const double t64 = S.d.t0 + ((double)(step0 + n) + c.cst) * S.d.dt;  // stage time, formed in FP64
      RainRec<T> rr = {nullptr, nullptr, T(0)};
      if (rain_kind == 3) {
        rr = rain_records<T>(S, t64);
        rr.r0 -= S.elem_begin;
        rr.r1 -= S.elem_begin;
      }
      Storm<T> storm = {};
      if constexpr (storm_regs<P, FT>()) storm = storm_at<T>(S, t64);
      const Acc zero = acc_make<Acc>(0.f, 0.f, 0.0);
      Acc rain_acc = zero, bdry_acc = zero;
      Elem<P, Pol> O;
      tile_body<P, FLUX, Pol, FT, true>(a, S, t64, rain_kind, press, rr, storm, tile, lane, valid, meta.z, meta.w,
                                        Wm + SL::REC + c.in * SL::RECS, halo, Wm + SL::GEO,
                                        reinterpret_cast<const unsigned*>(Wm + SL::PLAN),
                                        reinterpret_cast<const float*>(Wm + L::S_MAN),
                                        reinterpret_cast<const T*>(Wm + SL::XY), Wm + SL::FLX, Wm + SL::REC, s_ephi,
                                        s_ephi4, halo_ready,
                                        [&](bool mine, uint32_t at) {
                                          if (mine) {
                                            const uint32_t from = remote(at) + rin;
#pragma unroll
                                            for (int v = 0; v < RV; ++v)
                                              halo[v * HALO + lane] = ld_cluster128(from + 16u * TILE * v);
                                          }
                                          __syncwarp();
                                        },
                                        [] {},
                                        O, rain_acc, bdry_acc);
      if (valid) {
        Raw<RV> ro;
        pack<P>(O, ro);
        uint4* to = Wm + SL::REC + c.out * SL::RECS;
#pragma unroll
        for (int v = 0; v < RV; ++v) to[v * TILE + lane] = ro.v[v];
      }
      __syncwarp();
      cluster_arrive();
      // the stage's volume rates with its weight in the step; equal weights (SSP(2,2), SSP(5,2)) come at the
      // end of the launch
      if (!st.same_bw) {
        const Acc bw = acc_make<Acc>(c.bw_hi, c.bw_lo, c.bw);
        rain_acc = acc_mul(rain_acc, bw);
        bdry_acc = acc_mul(bdry_acc, bw);
      }
      long_add(rain_sum, rain_acc);
      long_add(bdry_sum, bdry_acc);
    }
  }
  cluster_wait();  // no CTA leaves while another reads its records
  if (present > 0) {
    if (valid) {
#pragma unroll
      for (int v = 0; v < RV; ++v) a.out[rec_at<RV>(tile * TILE + lane, v)] = Wm[SL::REC + v * TILE + lane];
    }
    double rain = long_d(rain_sum), bdry = long_d(bdry_sum);
    warp_reduce2(rain, bdry);
    if (lane == 0) {
      double* Lg = a.ledger + 2 * ((long long)sc * a.wslots + tile);
      const double wdt = st.same_bw ? st.st[0].bw * S.dt : S.dt;
      Lg[0] += wdt * rain;
      Lg[1] += wdt * bdry;
    }
  }
  if (blockIdx.x == 0 && tid == 0) a.ctl->step = step0 + st.nsteps;  // every CTA has read it: the barriers passed
}

// launch of one cluster of `ctas` CTAs, and whether such a launch can run on the device.  The
// kernel's shared-memory limit is raised to what the device allows, whatever this launch needs:
// several contexts with meshes of different sizes share the attribute.
template <int P, int FLUX, class Pol, int FT>
void steps_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* at, int ctas, int wpc, int nrec, cudaStream_t s) {
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim = {(unsigned)ctas, 1, 1};
  cfg = {};
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(32 * wpc);
  cfg.dynamicSmemBytes = steps_smem_per_warp<P, Pol, FT>(nrec) * wpc;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
}
template <int P, int FLUX, class Pol, int FT>
bool steps_fit_one(int ctas, int wpc, int nrec) {
  auto k = steps_kernel<P, FLUX, Pol, FT>;
  int dev = 0, optin = 0, n = 0;
  cudaFuncAttributes fa;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[1];
  steps_config<P, FLUX, Pol, FT>(cfg, at, ctas, wpc, nrec, nullptr);
  const bool ok = cudaGetDevice(&dev) == cudaSuccess &&
                  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) == cudaSuccess &&
                  cudaFuncGetAttributes(&fa, k) == cudaSuccess && 32 * wpc <= fa.maxThreadsPerBlock &&
                  (int)cfg.dynamicSmemBytes <= optin - (int)fa.sharedSizeBytes &&
                  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes) == cudaSuccess &&
                  cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                  cudaOccupancyMaxActiveClusters(&n, k, &cfg) == cudaSuccess && n >= 1;
  if (!ok) cudaGetLastError();
  return ok;
}
template <int P, int FLUX, class Pol, int FT>
cudaError_t steps_launch_one(const StageArgs<Pol>& a, const StepsArgs& st, int ctas, int wpc, cudaStream_t s) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[1];
  steps_config<P, FLUX, Pol, FT>(cfg, at, ctas, wpc, st.nrec, s);
  return cudaLaunchKernelEx(&cfg, steps_kernel<P, FLUX, Pol, FT>, a, st);
}

}  // namespace dg
