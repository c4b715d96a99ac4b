// Internal declarations shared by the libpf translation units.
#pragma once

#include <cuda_runtime.h>

#include "pf_common.cuh"

namespace pf {

// record the thread-local error message returned by pf_last_error; returns code
int set_error(int code, const char *msg);

// kernel-launch accounting (pf_launch_count)
void count_launches(long long n);

// supported tile shapes of the step kernels
struct TileShape {
    int tx, ty;
};

// 2D fused step (mode 0) or macroscopic-field pass (mode 1).  Returns false
// when the (precision, tile, moving, mode) combination is not compiled.
bool launch_step2d(int prec, int tx, int ty, bool moving, int mode, int grid, cudaStream_t s,
                   const StepArgs &a);
// query of the resident CTAs per SM of one 2D configuration (0 if unsupported)
int occupancy_step2d(int prec, int tx, int ty, bool moving, int mode);
bool launch_step2d_p64(int tx, int ty, bool moving, int mode, int grid, cudaStream_t s, const StepArgs &a, int *occ);
bool launch_step2d_p32(int tx, int ty, bool moving, int mode, int grid, cudaStream_t s, const StepArgs &a, int *occ);
bool launch_step2d_mixh(int tx, int ty, bool moving, int mode, int grid, cudaStream_t s, const StepArgs &a, int *occ);
bool launch_step2d_mixb(int tx, int ty, bool moving, int mode, int grid, cudaStream_t s, const StepArgs &a, int *occ);

// 3D: a tile marches through chunks of at most ZCHUNK3D planes in z
constexpr int ZCHUNK3D = 32;
bool launch_step3d(int prec, int tx, int ty, bool moving, int mode, int grid, cudaStream_t s,
                   const StepArgs &a);
int occupancy_step3d(int prec, int tx, int ty, bool moving, int mode);
void tile_shape3d(int prec, int *tx, int *ty);
bool launch_step3d_p64(int tx, int ty, bool moving, int mode, int grid, cudaStream_t s, const StepArgs &a, int *occ);
bool launch_step3d_p32(int tx, int ty, bool moving, int mode, int grid, cudaStream_t s, const StepArgs &a, int *occ);
bool launch_step3d_mixh(int tx, int ty, bool moving, int mode, int grid, cudaStream_t s, const StepArgs &a, int *occ);
bool launch_step3d_mixb(int tx, int ty, bool moving, int mode, int grid, cudaStream_t s, const StepArgs &a, int *occ);

void launch_init(int prec, const DomainDev &Dm, int *flags, const double *phi0, const double *phi, const double *u,
                 const double *Pin, double *tmp, const ParticleDev *parts, int np, int wv, cudaStream_t s);
int diag_blocks();
// Launch with programmatic dependence on the kernel before it in the stream (the
// kernel waits for it itself, see pdl_begin).  Per step in a graph, without and
// with: 250 x 223 (FP32) 5.85 and 5.45 us, the strip step of 1024^2 between walls (with
// the queue's memset gone) 51.1 and 47.7, 16 particles in 512^2 (step, repulsion and
// update) 39.4 and about 36.
template <class... K, class... A>
inline void launch_pdl(void (*kern)(K...), int grid, int threads, int dyn, cudaStream_t s, const A &...args)
{
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(grid);
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = dyn;
    c.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    c.attrs = at;
    c.numAttrs = 1;
    cudaLaunchKernelEx(&c, kern, args...);  // (its error is the launch's: cudaGetLastError)
}

void launch_diag(const DomainDev &Dm, double *scratch, const int *flags, int wv, cudaStream_t s);
// near / far tile lists of a particle domain (single-cell / two-cells step)
void launch_split_tiles(const StepArgs &a, int tx, int ty, unsigned char *sel, cudaStream_t s);
// interface normal (dim planes of N) from Dm.macro's phi plane
void launch_normal(const DomainDev &Dm, double *n, cudaStream_t s);
void launch_particle_update(ParticleDev *parts, int np, const double *partials, int ntiles,
                            const DevParams &p, double *frep, int nx, int ny, int nz, int wall_y,
                            const unsigned char *sel, cudaStream_t s);

}  // namespace pf
