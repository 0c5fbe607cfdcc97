#pragma once

#include "common.cuh"

namespace emsurf {

struct SlabType {
    long long offL[2];   // region v's L in the table buffer; its K follows at + E_v^2
    int Ev[2];
    int N, nint;
    long long offB;      // this type's N x N matrix in the elimination buffer
    long long offMap;    // this type's copy/sign arrays ([2][N])
};

// Eliminates the interior unknowns (the first nint of N) of every type's matrix
// in place: its trailing (N - nint) block becomes the Schur complement.  work:
// slab_lu_bytes of device memory; *status: 1 singular interior block, 2 expired wait.
size_t slab_lu_bytes(int types, int max_n, int max_nint);
int slab_lu(const SlabType* ty, int types, int max_n, int max_nint, double2* B, void* work, int* status, cudaStream_t st);

}  // namespace emsurf
