// Host-side interface of the ERI kernels (internal to the library).
#pragma once
#include <cuda_runtime.h>
#include "hfx_internal.cuh"

namespace hfx {

struct EriLaunch;

// Group sizes (lanes per quartet): 1 (a thread) or 32 (a warp).  Precision passes `prec`:
// 0 every quartet in FP64; 1 and 2 the FP64 and FP32 shares of a mixed-precision class.
// the default of a build of one system (uncontracted: every shell has one primitive), of all others 32
int eri_group_size(int cls, bool uncontracted, long long n_quartets, int n_sm);
bool eri_group_size_valid(int gs);
cudaError_t eri_prepare();
int eri_blocks_per_sm(int cls, int mode, int gs, int prec, bool batch);
// Streams (see hfx_set_streams; no kernel depends on them): the value reported for a choice
// (0 = the class default); whether a class has it.
int eri_streams(int cls, int streams);
bool eri_streams_valid(int cls, int streams);
// independent workers (threads, warps or teams of warps) of a block
int eri_groups_per_block(int cls, int gs);
// quartets per claim of the dynamic schedule, for a list of n_quartets and n_groups groups
int eri_chunk(int gs, long long n_quartets, long long n_groups);
// whether the next class launch may overlap this one
bool eri_overlap(int gs, long long n_quartets, long long n_groups);

// The Hermite engine (quartets on whole warps, hfx_md.cuh; f32: the FP32 pass) and its pair data.
// Kinds of launch: one system, a batch of systems, a lattice sum, the Schwarz diagonal.
enum { MD_PLAIN = 0, MD_BATCH = 1, MD_PER = 2, MD_DIAG = 3 };
size_t md_smem_bytes(int cls, bool f32);
cudaError_t md_prepare();
int md_blocks_per_sm(int cls, int kind, bool f32);
int md_teams_per_block(int cls);
cudaError_t md_launch(const EriLaunch& L, int cls, int kind, int prec, bool f32, int grid, cudaStream_t stream,
                      bool overlap);
cudaError_t launch_md_size(int n, const int* pcls, const int* cap, long long* size, cudaStream_t s);
cudaError_t launch_md_fill(int n, const int* pcls, const double* AB, const int* pp_off, const int* pp_n,
                           const PrimPair* pp, const long long* md_off, int hexp, double* md, cudaStream_t s);

}  // namespace hfx

namespace hfx {
// overlap: the launch before it on the stream is another class or pass of the same build, and this
// one need not wait for it (warps; the thread kernel always waits)
cudaError_t eri_launch(const EriLaunch& L, int cls, int mode, int grid, cudaStream_t stream, int gs, int prec,
                       bool batch, bool overlap = false);
}
