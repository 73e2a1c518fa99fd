// Host-side interface of the ERI kernels (internal to the library).
#pragma once
#include <cuda_runtime.h>
#include "hfx_internal.cuh"

namespace hfx {

struct EriLaunch;

// Group sizes (lanes per quartet): 1 (a thread) or 32 (a warp).  Precision passes `prec`:
// 0 every quartet in FP64; 1 and 2 the FP64 and FP32 shares of a mixed-precision class.
int eri_group_size();  // the default: 32
bool eri_group_size_valid(int gs);
size_t eri_smem_bytes(int cls, int gs, int streams = 0, int prec = 0);
cudaError_t eri_prepare();
int eri_blocks_per_sm(int cls, int mode, int gs, int prec, bool batch, int streams = 0);
// Streams of the warp kernel (primitive quartets run at a time): 0 = the class default;
// the value a launch with `streams` uses; whether a class has that variant.
int eri_streams(int cls, int streams);
bool eri_streams_valid(int cls, int streams);
// independent workers (threads, warps or teams of warps) of a block
int eri_groups_per_block(int cls, int gs, int prec);
// quartets per claim of the dynamic schedule, for a list of n_quartets and n_groups groups
int eri_chunk(int gs, long long n_quartets, long long n_groups);

// The Hermite engine (FP64 quartets on whole warps, hfx_md.cuh) and its pair data.
// Kinds of launch: one system, a batch of systems, a lattice sum, the Schwarz diagonal.
enum { MD_PLAIN = 0, MD_BATCH = 1, MD_PER = 2, MD_DIAG = 3 };
size_t md_smem_bytes(int cls);
cudaError_t md_prepare();
int md_blocks_per_sm(int cls, int kind);
int md_teams_per_block(int cls);
cudaError_t md_launch(const EriLaunch& L, int cls, int kind, int prec, int grid, cudaStream_t stream);
cudaError_t launch_md_size(int n, const int* pcls, const int* cap, long long* size, cudaStream_t s);
cudaError_t launch_md_fill(int n, const int* pcls, const double* AB, const int* pp_off, const int* pp_n,
                           const PrimPair* pp, const long long* md_off, double* md, cudaStream_t s);

}  // namespace hfx

namespace hfx {
cudaError_t eri_launch(const EriLaunch& L, int cls, int mode, int grid, cudaStream_t stream, int gs, int prec,
                       bool batch, int streams = 0);
}
