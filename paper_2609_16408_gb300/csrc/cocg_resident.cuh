// Resident COCG: one thread-block cluster runs the whole COCG loop of one Sternheimer system.
#pragma once
#include "cocg.cuh"

namespace rpa {

constexpr int kResMaxCluster = 16;
constexpr int kTileResident = -7;  // rpa_stats.tile_rows of loops that this kernel runs
// How a grid is cut over the blocks of a cluster, and what the launch needs.
struct ResidentShape {
  int G = 0;          // blocks of a cluster (0: the grid does not fit)
  int gy = 1, gz = 1; // the y and z extents are cut into gy x gz bricks of full x rows
  int bym = 0, bzm = 0;  // largest brick
  int pitch = 0;      // row pitch in shared memory (odd: rows of one column fall in distinct banks)
  int lx = 0, ly = 0, lz = 0;  // outputs of a thread's segment of a grid line, per axis
  int r_res = 0, x_res = 0;    // r and x in shared memory too (else in global memory)
  int threads = 0;
  size_t smem = 0;
  int clusters = 0;   // clusters the GPU holds at a time
};

// 32-entry steps whose loads a warp has in flight at a time
template <typename T>
__host__ __device__ constexpr int res_steps() {
  return sizeof(T) == 4 ? 8 : 4;
}
// Projector entries as the warps of a cluster read them, 32 (a step) at a time; slots are
// shared-memory slots of the entry's brick.
//   for chi^T p: records of up to res_steps() steps of one group, dealt to the warps in turn;
//     the records of a group follow one another
//   for w += chi cp: a warp owns a run of slots and takes their entries in layers of distinct
//     slots, so that no two warps, and no two lanes of a step, touch the same point
template <typename T>
struct ResidentProj {
  int ngroup = 0;
  const T* coef = nullptr;                // ngroup x 4: gamma dV
  const int* roff = nullptr;              // G + 1: first record of each block
  const int* rstep = nullptr;             // records + 1: first step of each record
  const unsigned short* gslot = nullptr;  // 32 per step (padding: slot 0, zero values)
  const T* gchi = nullptr;                // 4 per entry
  const int* goff = nullptr;              // G + 1: offsets into groups
  const int* groups = nullptr;            // (group, first record, end record) of a block
  const int* lwarp = nullptr;             // G * warps + 1: first step of each warp
  const unsigned* lkey = nullptr;         // group << 16 | slot (padding: all ones)
  const T* lchi = nullptr;
  const unsigned* gmask = nullptr;        // per group: the blocks with entries of it
};

// out[i] = the four values of entry e[i], zeros where e[i] < 0
template <typename T>
cudaError_t resident_gather(long long n, const int* e, const T* chi, T* out, cudaStream_t s);

bool resident_supported(int R);
// Shape for a grid of nx x ny x nz points and clusters of G blocks (G = 0 in the result if it
// does not fit).
template <typename T>
cudaError_t resident_shape(int nx, int ny, int nz, int R, int ngroup, int G, ResidentShape* out);
// COCG loop of every active system of cv: x, r (and, with cont, the direction kept in cv.p and
// beta) as for the fused iteration; on return x is the solution, cv.p the last direction of
// the systems that ran an even number of iterations since their kIterBase, p_odd (may be null)
// that of the others, and sysd / sysi hold the status, iterations and rho.
template <typename T>
cudaError_t resident_cocg(const CocgView<T>& cv, const ResidentShape& sh,
                          const ResidentProj<T>& pj, cpx<T>* p_odd, int maxit, int cont,
                          cudaStream_t s);

}  // namespace rpa
