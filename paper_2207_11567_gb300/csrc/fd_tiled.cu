// Host side of the tiled FD update (fd_tiled.cuh): eligibility, TMA tensor maps, launch.
#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <new>
#include <vector>
#include "fd_tiled.cuh"
#include "launch.h"

namespace hlbm {

namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)p;
  }
  return fn;
}

// Tensor over (x, y, z[, comp]) of a [comps][nz][ny][nx] array, box (40, 12, 1[, comps]).
bool make_map(CUtensorMap* m, CUtensorMapDataType dt, const void* base, const Geo& g, int comps) {
  const int rank = comps > 1 ? 4 : 3;
  cuuint64_t dims[4] = {(cuuint64_t)g.nx, (cuuint64_t)g.ny, (cuuint64_t)g.nz, (cuuint64_t)comps};
  cuuint64_t strides[3] = {(cuuint64_t)g.nx * 4, (cuuint64_t)g.nx * g.ny * 4, (cuuint64_t)g.N * 4};
  cuuint32_t box[4] = {(cuuint32_t)TT_PX, (cuuint32_t)TT_PY, 1u, (cuuint32_t)comps};
  cuuint32_t es[4] = {1, 1, 1, 1};
  const CUresult r = encode_fn()(m, dt, (cuuint32_t)rank, const_cast<void*>(base), dims, strides, box, es,
                                 CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                 CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

template <int NK, int NR> cudaError_t set_smem() {
  return cudaFuncSetAttribute(fd_tiled_kernel<NK, NR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)TTLayout<NK>::BYTES);
}

}  // namespace

bool fd_tiled_eligible(const Geo& g, int D, int f64, int varcp, int K, int nrx) {
  if (D != 3 || f64 || varcp) return false;
  if (!((K == 6 && nrx == 2) || (K == 4 && nrx == 1))) return false;
  for (int a = 0; a < 3; ++a)
    if (g.bc_lo[a] == BC_PERIODIC || g.bc_hi[a] == BC_PERIODIC) return false;
  if (g.nx % 4 != 0) return false;  // TMA: row strides are multiples of 16 bytes
  return encode_fn() != nullptr;
}

FDTiledMaps* fd_tiled_create() { return new (std::nothrow) FDTiledMaps(); }
void fd_tiled_destroy(FDTiledMaps* m) { delete m; }

cudaError_t fd_tiled_setup(FDTiledMaps& m, const Geo& g, int K, void* const T[2], void* const Y[2],
                           void* const F[2], const void* u, const uint32_t* sword, int n_sm) {
  m.sensor = F[0] != nullptr;
  bool ok = true;
  for (int b = 0; b < 2; ++b) {
    ok = ok && make_map(&m.T[b], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, T[b], g, 1);
    ok = ok && make_map(&m.Y[b], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, Y[b], g, K);
    m.F[b] = m.T[b];
    if (m.sensor) ok = ok && make_map(&m.F[b], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, F[b], g, 1);
  }
  ok = ok && make_map(&m.U, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, u, g, 3);
  ok = ok && make_map(&m.S, CU_TENSOR_MAP_DATA_TYPE_UINT32, sword, g, 1);
  if (!ok) return cudaErrorInvalidValue;
  m.gx = (g.nx + TT_X - 1) / TT_X;
  m.gy = (g.ny + TT_Y - 1) / TT_Y;
  m.slots = 2 * n_sm;
  cudaError_t e = set_smem<6, 2>();
  if (e == cudaSuccess) e = set_smem<4, 1>();
  return e;
}

int fd_tiled_tiles(const FDTiledMaps& m, const Geo& g) { return m.gx * m.gy * ((g.nz + TT_LZ_MIN - 1) / TT_LZ_MIN); }

int fd_tiled_blocks(const FDTiledMaps& m) { return m.n_tiles; }

// The tiles to launch: those with a fluid cell (swirl burner, all tiles / these: 384x192x192, where 22% of
// the cells are solid, 759 / 698 us per update, 192x96x96 150.2 / 147.5), for the number of planes per
// tile that costs least: whole waves of the resident blocks (two per SM), each as long as its planes plus
// about three for the block's start (its first three plane loads and the -z face). Planes per tile, update
// of 384x192x192: 6 733 us, 8 718, 12 708, 16 709, 24 716; of 192x96x96 with curved walls: 6 166, 8 163.5,
// 12 162.3, 16 183.8 (one wave and a short second one).
cudaError_t fd_tiled_set_mask(FDTiledMaps& m, const Geo& g, const uint8_t* mask, int* tiles_dev, cudaStream_t st) {
  const size_t cols = (size_t)m.gx * m.gy;
  std::vector<uint8_t> live(cols * g.nz, 0);  // per plane
  for (int z = 0; z < g.nz; ++z)
    for (int y = 0; y < g.ny; ++y) {
      const uint8_t* row = mask + (size_t)g.nx * (y + (size_t)g.ny * z);
      uint8_t* l = live.data() + cols * z + (size_t)m.gx * (y / TT_Y);
      for (int t = 0; t < m.gx; ++t)
        if (!l[t] && std::memchr(row + t * TT_X, 0, std::min(TT_X, g.nx - t * TT_X))) l[t] = 1;
    }
  auto tiles_of = [&](int lz) {
    std::vector<int> list;
    for (int z0 = 0, k = 0; z0 < g.nz; z0 += lz, ++k)
      for (size_t t = 0; t < cols; ++t) {
        bool any = false;
        for (int z = z0; z < std::min(z0 + lz, g.nz) && !any; ++z) any = live[cols * z + t] != 0;
        if (any) list.push_back((int)(t + cols * k));
      }
    return list;
  };
  std::vector<int> list;
  double best = 1e30;
  for (int lz = std::min(TT_LZ_MIN, g.nz); lz <= std::min(g.nz, TT_LZ_MAX); ++lz) {
    std::vector<int> l = tiles_of(lz);
    const double cost = (double)(((int)l.size() + m.slots - 1) / m.slots) * (lz + 3);
    if (cost < best) {
      best = cost;
      m.lz = lz;
      list.swap(l);
    }
  }
  m.tiles = tiles_dev;
  m.n_tiles = (int)list.size();
  if (list.empty()) return cudaSuccess;
  const cudaError_t e = cudaMemcpyAsync(tiles_dev, list.data(), list.size() * sizeof(int), cudaMemcpyHostToDevice, st);
  return e == cudaSuccess ? cudaStreamSynchronize(st) : e;
}

namespace {
template <int NK, int NR>
cudaError_t launch_tiles(const FDArgs<float>& a, const FDTiledMaps& m, int cur, cudaStream_t st, bool pdl) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(m.n_tiles);
  cfg.blockDim = dim3(TT_X, TT_Y);
  cfg.dynamicSmemBytes = TTLayout<NK>::BYTES;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, fd_tiled_kernel<NK, NR>, a, m.T[cur], m.Y[cur], m.U, m.F[cur], m.S,
                            (const int*)m.tiles, m.lz, a.Floc ? 1 : 0);
}
}  // namespace

cudaError_t launch_fd_tiled(const FDArgs<float>& a, const FDTiledMaps& m, int cur, cudaStream_t st, bool pdl) {
  if (m.n_tiles == 0) return cudaSuccess;
  return a.c.K == 6 && a.c.nrx == 2 ? launch_tiles<6, 2>(a, m, cur, st, pdl) : launch_tiles<4, 1>(a, m, cur, st, pdl);
}

}  // namespace hlbm
