// smerf_setup.h -- the set-up entry point (smerf_setup.cu) used by smerf_api.cu.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>

struct smerf_plan;

// Set-up of a plan's tables (Alg. 1), every device step ordered on `st`.  sync: wait for it
// and record setup_ms; otherwise the caller synchronises `st` before the plan is used.  held: the
// bytes of the scratch pool reserved for set-ups on this stream (smerf_setup_reserve), which the caller
// releases once the stream is synchronised.
int smerf_setup_tables(smerf_plan* plan, cudaStream_t st, bool sync, size_t* held);

// Set-ups' temporaries in the scratch pool, which keeps its memory: at most 512 MB of it over every set-up
// in flight (smerf_plan_create_many overlaps 16 of up to 256 MB).  smerf_setup_reserve raises a stream's
// share *held to `bytes` if that fits (a stream's set-ups follow each other and take the same memory);
// otherwise the caller takes the default pool, which returns its memory.
bool smerf_setup_reserve(size_t bytes, size_t* held);
void smerf_setup_release(size_t held);

// Whether the ring colatitudes (n_theta values, increasing) are symmetric about the equator,
// theta_k + theta_{n_theta-1-k} = pi within 1e-12 pi; NULL (the equiangular grid) is.  On a
// symmetric grid the southern chain's steps are the northern ones mirrored and the start ring is
// n_theta / 2; otherwise the start ring is the ring nearest the equator and the southern chain's
// steps are computed on their own.
bool smerf_grid_symmetric(const double* theta, int n_theta);

// The start ring k0 of both chains (Alg. 2 starts at the equator): n_theta / 2 on a symmetric
// grid (the equator ring for odd n_theta, the first ring south of it for even n_theta), else the
// ring whose colatitude is nearest pi / 2, the southern one of two at the same distance.
int smerf_start_ring(const double* theta, int n_theta);
