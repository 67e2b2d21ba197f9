// Launches of the V-cycle legs of leg_device.cuh on one device stack.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>

#include "ferrox_internal.cuh"
#include "leg_device.cuh"

namespace fx {

namespace {

using namespace dev;

template <int TX, int TY, bool SC, bool CONT>
__global__ void __launch_bounds__(LegDown<TX, TY, SC, CONT>::G::THREADS, leg_min_blocks(LegDown<TX, TY, SC, CONT>::G::THREADS, SC)) leg_down_kernel(LegArgs a) {
  extern __shared__ __align__(16) unsigned char leg_smem[];
  pdl_enter();
  LegDown<TX, TY, SC, CONT>::run(a, blockIdx.x, blockIdx.y, blockIdx.z, leg_smem);
}

template <int TX, int TY, bool SC, bool PHI>
__global__ void __launch_bounds__(LegUp<TX, TY, SC, PHI>::G::THREADS, leg_min_blocks(LegUp<TX, TY, SC, PHI>::G::THREADS, SC || PHI)) leg_up_kernel(LegArgs a, Upd u, const DevStats* st) {
  extern __shared__ __align__(16) unsigned char leg_smem[];
  pdl_enter();
  if (PHI) u.zero = st->zero_phi;
  LegUp<TX, TY, SC, PHI>::run(a, u, blockIdx.x, blockIdx.y, blockIdx.z, leg_smem);
}

template <int TX, int TY>
dim3 leg_grid(const LegArgs& a) {
  return dim3((a.nx + TX - 1) / TX, (a.ny + TY - 1) / TY, (a.nz + a.kz - 1) / a.kz);
}

template <int TX, int TY, bool SC, bool CONT>
void down(const LegArgs& a, cudaStream_t s) {
  using K = LegDown<TX, TY, SC, CONT>;
  launch_k(leg_down_kernel<TX, TY, SC, CONT>, leg_grid<TX, TY>(a), dim3(K::G::THREADS), K::smem_bytes(a.kz), s, a);
}

template <int TX, int TY, bool SC, bool PHI>
void up(const LegArgs& a, const UpdateArgs* upd, cudaStream_t s) {
  using K = LegUp<TX, TY, SC, PHI>;
  Upd u{nullptr, 0.0, 0, 0.0f};
  const DevStats* st = nullptr;
  if (upd) { u.phi = upd->phi; u.clamp = upd->clamp; u.clampf = (float)upd->clamp; st = upd->stats; }
  launch_k(leg_up_kernel<TX, TY, SC, PHI>, leg_grid<TX, TY>(a), dim3(K::G::THREADS), K::smem_bytes(a.kz), s, a, u, st);
}

cudaError_t allow_smem(const void* f) {
  return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
}

template <int TX, int TY>
cudaError_t prepare_tile() {
  for (const void* f : {(const void*)leg_down_kernel<TX, TY, false, false>, (const void*)leg_down_kernel<TX, TY, false, true>,
                        (const void*)leg_down_kernel<TX, TY, true, false>, (const void*)leg_down_kernel<TX, TY, true, true>,
                        (const void*)leg_up_kernel<TX, TY, false, false>, (const void*)leg_up_kernel<TX, TY, false, true>,
                        (const void*)leg_up_kernel<TX, TY, true, false>, (const void*)leg_up_kernel<TX, TY, true, true>})
    if (const cudaError_t e = allow_smem(f); e != cudaSuccess) return e;
  return cudaSuccess;
}

template <int TX, int TY>
void down_tile(const LegArgs& a, cudaStream_t s) {
  if (a.s) a.e_in ? down<TX, TY, true, true>(a, s) : down<TX, TY, true, false>(a, s);
  else a.e_in ? down<TX, TY, false, true>(a, s) : down<TX, TY, false, false>(a, s);
}

template <int TX, int TY>
void up_tile(const LegArgs& a, const UpdateArgs* upd, cudaStream_t s) {
  if (a.s) upd ? up<TX, TY, true, true>(a, upd, s) : up<TX, TY, true, false>(a, upd, s);
  else upd ? up<TX, TY, false, true>(a, upd, s) : up<TX, TY, false, false>(a, upd, s);
}

}  // namespace

// Tile and planes per block by the level's size, from the legs timed one by one in a
// graph (us, down / up; tile/kz): small levels want blocks on every SM more than they
// mind the recomputed halo,
//   32x32x4      16x16/2 2.9 / 4.4, 32x16/4 3.4 / 4.7        64x64x8  16x16/2 3.5 / 5.6, 32x16/4 4.4 / 6.5
//   128x128x16   32x16/4 4.6 / 7.5, 16x16/4 5.2 / 7.7, 32x16/16 6.6 / 9.7,
// large ones the smaller halo share of long columns,
//   256x256x32   32x16/32 11.4 / 18.0, 32x16/16 12.3 / 16.8, 32x16/8 15.5 / 22.8
//   512x512x128 (shift)  32x16/128 297 / 217, 32x16/32 287 / 232, 32x16/16 325 / 281,
// and with a shift the down leg that continues a correction (six registers more per
// cell) the larger tile: 256x256x64 32x32/32 37, 32x16/32 50.
// An up leg whose blocks would leave SMs idle takes 16 planes, two blocks to an SM (its
// phi update waits on memory): 256x256x32, 256 blocks instead of 128: both fine legs, timed one
// by one, 52 -> 45.5 us; the down leg gains nothing from it, and 256x256x64 (256 blocks
// of 32 planes) loses.
LegPlan leg_plan(long long cells, int nx, int ny, int nz, bool wide, bool up) {
  if (cells < (1 << 17)) return {kLegTile16x16, 2};
  if (cells < (1 << 20)) return {kLegTile32x16, 4};
  const long long tiles = (long long)((nx + 31) / 32) * ((ny + 15) / 16);
  int kz = 32;
  while (kz < 128 && tiles * ((nz + kz - 1) / kz) > 600) kz *= 2;
  if (up && tiles * ((nz + kz - 1) / kz) < 152) kz = 16;
  return {wide ? kLegTile32x32 : kLegTile32x16, kz};
}

bool leg_level(const LevelDesc& L) { return L.crx && L.cry && !(L.nx & 1) && !(L.ny & 1); }

cudaError_t leg_prepare() {
  cudaError_t e;
  if ((e = allow_smem((const void*)leg_down_kernel<32, 32, true, true>)) != cudaSuccess) return e;
  if ((e = prepare_tile<32, 16>()) != cudaSuccess) return e;
  return prepare_tile<16, 16>();
}

void launch_leg_down(const LegArgs& a_in, cudaStream_t s) {
  LegArgs a = a_in;
  const LegPlan p = leg_plan((long long)a.nx * a.ny * a.nz, a.nx, a.ny, a.nz, a.s && a.e_in);
  a.kz = std::min(p.kz, a.nz + (a.nz & 1));
  if (p.tile == kLegTile32x32) down<32, 32, true, true>(a, s);   // wide levels only
  else if (p.tile == kLegTile32x16) down_tile<32, 16>(a, s);
  else down_tile<16, 16>(a, s);
}

void launch_leg_up(const LegArgs& a_in, const UpdateArgs* upd, cudaStream_t s) {
  LegArgs a = a_in;
  const LegPlan p = leg_plan((long long)a.nx * a.ny * a.nz, a.nx, a.ny, a.nz, false, true);
  a.kz = std::min(p.kz, a.nz + (a.nz & 1));
  a.phi_vec = upd && reinterpret_cast<uintptr_t>(upd->phi) % 16 == 0;
  if (p.tile == kLegTile32x16) up_tile<32, 16>(a, upd, s);
  else up_tile<16, 16>(a, upd, s);
}

}  // namespace fx
