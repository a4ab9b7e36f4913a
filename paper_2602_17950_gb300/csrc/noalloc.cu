// Allocation-free variant of gpsoc_apply_h.
//
// Some callers cannot allocate device memory at the point where they need the
// Hamiltonian: a host framework that has already handed all device memory to its
// own pool, a real-time loop that must not pay for (or synchronise on)
// cudaMalloc/cudaFree, or code running under a fixed memory budget that has been
// reserved up front.  gpsoc_apply_h_noalloc serves them: it takes the wave
// functions and the output buffer from the caller and keeps every intermediate
// array, partial sum, twiddle table and per-solve scalar in one file-scope device
// array of fixed size, kNoAllocScratchBytes, that exists once per GPU from the
// moment the library is loaded until the process exits.
//
// Nothing here allocates: no cudaMalloc, cudaFree, cudaMallocHost or host heap
// (failures are reported through the returned status only; gpsoc_last_error
// is not updated by this call).
// The device address of the array is looked up once per device with
// cudaGetSymbolAddress (the host-side name of a __device__ array is only a
// stand-in and must never be handed to a kernel).
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <mutex>

#include "gpsoc_internal.cuh"
#include "kernels.cuh"

using namespace gpsoc;

static constexpr size_t kNoAllocScratchBytes = 16u << 20;   // 16 MiB per device

// the scratch of every call; in host code this name is a stand-in, not a device address
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

namespace {

constexpr int kMaxDevices = 64;

unsigned char* g_scratch_ptr[kMaxDevices] = {};
std::mutex g_scratch_mu;

// device address of the scratch array on the current device (set up on first use)
cudaError_t scratch_address(unsigned char** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(g_scratch_mu);
  if (!g_scratch_ptr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return e;
    e = chain_prepare<double>();   // kernel attributes (idempotent)
    if (e != cudaSuccess) return e;
    g_scratch_ptr[dev] = (unsigned char*)p;
  }
  *out = g_scratch_ptr[dev];
  return cudaSuccess;
}

__host__ __device__ void put_obs(const SolveState& S, double* o) {
  o[0] = S.E; o[1] = S.mu;
  for (int c = 0; c < 3; ++c) { o[2 + c] = S.alpha[c]; o[5 + c] = S.mass[c]; }
  o[8] = S.Q;
}

__global__ void k_gather_obs(const SolveState* st, int batch, double* out) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= batch) return;
  put_obs(st[s], out + 9 * s);
}

// parameters (in the launch's own argument space: no copy from the host), cleared states and arrival counters.
// With the observables taken in the last block of the last pass and small batches' states read whole, a
// call is 4 launches and a copy instead of 6 launches and 4 copies: 73.4 -> 69.6 us for one 64^2 solve
constexpr int kSetup = 64;   // solves per launch
struct SetupParams { PhysDev p[kSetup]; };
__global__ void k_setup(SolveState* st, unsigned* cnt, PhysDev* phys, SetupParams q, int first, int count,
                        int counters) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= count) return;
  SolveState z{};
  z.active = 1;
  st[first + k] = z;
  for (int i = 0; i < counters; ++i) cnt[(first + k) * counters + i] = 0u;
  phys[first + k] = q.p[k];
}

// What a state and a point of an axis count in the budget.  They are the sizes of an earlier layout (a larger state, a
// twiddle table per axis) and stay what they were, so that a request that fitted still fits; the arrival
// counters lie in the axes' share.
constexpr size_t kStateBudget = 488, kAxisBudget = 16;
static_assert(sizeof(SolveState) <= kStateBudget, "the budget of a state is part of the call's limit");

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

int ilog2i(int n) { int l = 0; while ((1 << l) < n) ++l; return l; }

}  // namespace

extern "C" gpsoc_status gpsoc_apply_h_noalloc(const gpsoc_grid* grid, const gpsoc_trap* trap,
                                              const gpsoc_params* params, int batch, const void* d_psi,
                                              void* d_hpsi, double* obs, void* cuda_stream) {
  if (!grid || !trap || !params || !d_psi || !d_hpsi || batch < 1) return GPSOC_EINVAL;
  if (grid->dim != 2 && grid->dim != 3) return GPSOC_EINVAL;
  // the same trap checks as gpsoc_create; user potentials would need device memory of their own
  if (trap->kind != GPSOC_TRAP_HARMONIC && trap->kind != GPSOC_TRAP_HARMONIC_QUARTIC) return GPSOC_EINVAL;
  for (int i = 0; i < grid->dim; ++i)
    if (!std::isfinite(trap->g[i])) return GPSOC_EINVAL;
  if (!std::isfinite(trap->quad) || !std::isfinite(trap->quart)) return GPSOC_EINVAL;
  Geo g{};
  g.d = grid->dim;
  g.npts = 1;
  g.dV = 1.0;
  for (int i = 0; i < 3; ++i) {
    if (i < grid->dim) {
      const int n = grid->n[i];
      if (n < 8 || n > 1024 || (n & (n - 1))) return GPSOC_EINVAL;
      if (!(grid->L[i] > 0) || !std::isfinite(grid->L[i])) return GPSOC_EINVAL;
      g.n[i] = n;
      g.L[i] = grid->L[i];
      g.h[i] = 2.0 * grid->L[i] / n;
      g.piL[i] = 3.14159265358979323846 / grid->L[i];
      g.dV *= g.h[i];
    } else {
      g.n[i] = 1; g.L[i] = 1.0; g.h[i] = 1.0; g.piL[i] = 0.0;
    }
    g.log2n[i] = ilog2i(g.n[i]);
    g.npts *= g.n[i];
  }
  // scratch layout: A, B, W, G arrays | partial sums | states | parameters | observables
  const size_t arr = sizeof(double2) * (size_t)batch * 3 * g.npts;
  const int nb_row = row_blocks_per_solve<double>(g, batch);
  int pmax = nb_row;
  for (int ax = 1; ax < g.d; ++ax) pmax = std::max(pmax, col_blocks_per_solve<double>(g, ax, batch));
  size_t off = 0;
  const size_t o_arr = off; off += align256(4 * arr);
  const size_t o_part = off; off += align256(sizeof(double) * (size_t)batch * NSLOT * pmax);
  const size_t o_st = off; off += align256(kStateBudget * batch);
  const size_t o_ph = off; off += align256(sizeof(PhysDev) * batch);
  const size_t o_cnt = off;
  for (int i = 0; i < g.d; ++i) off += align256(kAxisBudget * g.n[i]);
  const size_t o_obs = off; off += align256(sizeof(double) * 9 * batch);
  // a group counter per 64 blocks: 4 (1 + pmax / 64) bytes a solve of the axes' share and the observables' 72
  const int gmax = (pmax + 63) / 64;
  if (off > kNoAllocScratchBytes || sizeof(unsigned) * (size_t)batch * (1 + gmax) > off - o_cnt) return GPSOC_EBUDGET;
  // every check before the first launch: a call that returns an error leaves nothing running
  for (int k = 0; k < batch; ++k) {
    const gpsoc_params& r = params[k];
    if (!std::isfinite(r.Omega) || !std::isfinite(r.gamma) || !std::isfinite(r.beta0) || !std::isfinite(r.beta1))
      return GPSOC_EINVAL;
  }
  unsigned char* base = nullptr;
  cudaError_t e = scratch_address(&base);
  if (e != cudaSuccess) return GPSOC_ECUDA;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  double2* A = (double2*)(base + o_arr);
  double2* Bb = A + (size_t)batch * 3 * g.npts;
  double2* W = Bb + (size_t)batch * 3 * g.npts;
  double2* G = W + (size_t)batch * 3 * g.npts;
  double* part = (double*)(base + o_part);
  SolveState* sst = (SolveState*)(base + o_st);
  PhysDev* ph = (PhysDev*)(base + o_ph);
  double* dobs = (double*)(base + o_obs);
  // arrival counters of every solve's blocks and groups of 64 blocks: in the axes' share and, where many small
  // solves need it, on into the place of the gathered observables, which are written after the last arrival
  unsigned* cnt = (unsigned*)(base + o_cnt);
  for (int b0 = 0; b0 < batch; b0 += kSetup) {
    SetupParams q;
    const int nb = std::min(kSetup, batch - b0);
    for (int k = 0; k < nb; ++k) {
      const gpsoc_params& r = params[b0 + k];
      q.p[k] = make_phys(r.Omega, r.gamma, r.beta0, r.beta1);
    }
    k_setup<<<1, kSetup, 0, st>>>(sst, cnt, ph, q, b0, nb, 1 + gmax);
  }
  ChainArgs<double> a{};
  a.g = g;
  for (int i = 0; i < 3; ++i) a.trap.half_g2[i] = (i < g.d) ? 0.5 * trap->g[i] * trap->g[i] : 0.0;
  a.trap.quad = (trap->kind == GPSOC_TRAP_HARMONIC) ? 0.0 : trap->quad;
  a.trap.quart = (trap->kind == GPSOC_TRAP_HARMONIC) ? 0.0 : trap->quart;
  a.trap.userV = nullptr;
  a.phys = ph;
  a.st = sst;
  a.part = part;
  a.pmax = pmax;
  a.gate = GATE_ALL;
  a.nsolve = batch;
  a.scale = 1.0;
  a.cnt = cnt;
  a.gcnt = cnt + batch;
  a.gmax = gmax;
  // the Hamiltonian chain of gpsoc_apply_h, on the caller's buffers and the scratch
  const double2* src = (const double2*)d_psi;
  a.in0 = src; a.out0 = A;
  launch_row<double>(ROW_FWD_PLAIN, a, 0, Launch{}, st);
  if (g.d == 2) {
    a.in0 = A; a.out0 = W; a.out1 = G;
    launch_col<double>(COL_YMID_H, 1, a, Launch{}, st);
  } else {
    a.in0 = A; a.out0 = Bb; a.out1 = nullptr;
    launch_col<double>(COL_FWD, 1, a, Launch{}, st);
    a.in0 = Bb; a.out0 = Bb;
    launch_col<double>(COL_MID_H, 2, a, Launch{}, st);
    a.in0 = Bb; a.in1 = A; a.out0 = W; a.out1 = G;
    launch_col<double>(COL_YINV_H, 1, a, Launch{}, st);
  }
  // the last pass also takes E, mu, alpha and the masses from its sums
  a.in0 = W; a.in1 = G; a.in2 = src; a.out0 = (double2*)d_hpsi; a.out1 = nullptr;
  a.fuse = 1;
  a.sc.st = sst; a.sc.phys = ph; a.sc.part = part; a.sc.pmax = pmax;
  a.sc.nb_row = nb_row;
  a.sc.nb_col = col_blocks_per_solve<double>(g, g.d - 1, batch);
  a.sc.npts = g.npts; a.sc.dV = g.dV;
  a.sc.inv_npts = 1.0 / (double)g.npts;
  launch_row<double>(ROW_INV_H, a, 0, Launch{}, st);
  constexpr int kStates = 16;
  if (batch > kStates) k_gather_obs<<<(batch + 127) / 128, 128, 0, st>>>(sst, batch, dobs);
  e = cudaGetLastError();
  if (e != cudaSuccess) return GPSOC_ECUDA;
  // a few states are read whole and picked apart here, many are gathered first
  SolveState hst[kStates];
  if (obs) {
    e = batch > kStates ? cudaMemcpyAsync(obs, dobs, sizeof(double) * 9 * batch, cudaMemcpyDeviceToHost, st)
                        : cudaMemcpyAsync(hst, sst, sizeof(SolveState) * batch, cudaMemcpyDeviceToHost, st);
    if (e != cudaSuccess) return GPSOC_ECUDA;
  }
  e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return GPSOC_ECUDA;
  if (obs && batch <= kStates)
    for (int k = 0; k < batch; ++k) put_obs(hst[k], obs + 9 * k);
  return GPSOC_OK;
}
