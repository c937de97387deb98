// clot_eta_dct.cu -- the eta solve of meshes the direct solver takes
// (clot_eta_dct.cuh) as a launch of its own, and the solver's tables.
#include <algorithm>

#include "clot_eta_dct.cuh"

namespace clot {
namespace {

constexpr int DT = DCT_THREADS;

__global__ void __launch_bounds__(DT, 3) eta_dct_kernel(const __grid_constant__ EtaArgs a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  Team T{(int)gridDim.x, 0u, 0, true};
  EtaOut o;
  bool solved;
  const bool ok = eta_solve_team<DT>(a, *reinterpret_cast<DctSm*>(smraw), T, o, solved);
  if (!solved && ok) return;  // prediction accepted: no block arrived anywhere
  eta_note(a, o, ok);
  team_leave(a);
}

// The axis' matrices and eigenvalues (FP64 cosines, rounded once).
__global__ void dct_table_kernel(int n, int H, float* out) {
  const long long HH = (long long)H * H;
  const long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (x < 4 * HH) {
    const int mat = (int)(x / HH), par = mat & 1, row = (int)(x % HH / H), col = (int)(x % H);
    const int j = mat < 2 ? row : col, m = 2 * (mat < 2 ? col : row) + par;
    float v = 0.0f;
    if (m < n && j < (n + 1) / 2) {
      const long long ph = (long long)m * (2 * j + 1) % (4 * n);
      v = (float)(sqrt((m ? 2.0 : 1.0) / n) * cospi((double)ph / (2.0 * n)));
    }
    out[x] = v;
  } else if (x < 4 * HH + n) {
    const double s = sinpi((double)(x - 4 * HH) / (2.0 * n));
    out[x] = (float)(4.0 * s * s);
  }
}

}  // namespace

long long dct_table_floats(int n) {
  const long long H = dct_half(n);
  return 4 * H * H + (n + 3) / 4 * 4;
}

cudaError_t launch_dct_table(int n, float* out, cudaStream_t s) {
  const long long tot = dct_table_floats(n);
  dct_table_kernel<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(n, dct_half(n), out);
  return cudaGetLastError();
}

bool dct_applies(const Geom& g) { return g.nx <= DCT_MAX_NX && g.ny <= DCT_MAX_N && (g.dim == 2 || g.nz <= DCT_MAX_N); }

int dct_max_grid(const Geom& g) {
  int dev = 0, sms = 0, per_sm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  if (cudaFuncSetAttribute(eta_dct_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, sizeof(DctSm)) != cudaSuccess)
    return 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, eta_dct_kernel, DT, sizeof(DctSm)) != cudaSuccess) return 0;
  // at most a block per 32-mode tile of a whole-mesh pass, or per four mode lines
  const long long W4 = (g.nx + 3) / 4 * 4;
  auto tiles = [&](long long cols, int n) { return (cols / 4 + 15) / 16 * 2 * ((((long long)n + 1) / 2 + 31) / 32); };
  long long need = std::max(tiles(W4 * g.nz, g.ny), ((long long)g.ny * g.nz + DT / 32 - 1) / (DT / 32));
  if (g.dim == 3) need = std::max(need, tiles(W4 * g.ny, g.nz));
  return (int)std::min<long long>(need, (long long)sms * std::max(per_sm, 1));
}

cudaError_t launch_eta_dct(const EtaArgs& a, int grid, cudaStream_t s) {
  EtaArgs copy = a;
  void* args[] = {&copy};
  return cudaLaunchCooperativeKernel((const void*)eta_dct_kernel, dim3(grid), dim3(DT), args, sizeof(DctSm), s);
}

}  // namespace clot
