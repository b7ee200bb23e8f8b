// mrq_internal.h - what the runtime (mrq.cu) shares with the other translation units of the
// library: a read-only view of a context's loaded Hamiltonian and its error slot.  Not part of
// the C ABI.
#ifndef MRQ_INTERNAL_H
#define MRQ_INTERNAL_H

#include <cuda_runtime.h>

struct mrq_ctx;

struct MrqHamView {
    int device;
    cudaStream_t stream;
    int n, nc, na, nv, nalpha, nbeta, W;
    const double* h1;        // n x n row-major, device
    const double* eri;       // 8-fold packed (pq|rs), device
    long long neri;
    double e_nuc;
};

// MRQ_NOT_LOADED (message set) when the context holds no Hamiltonian
int mrq_internal_ham(mrq_ctx* ctx, MrqHamView* out);
// record a message in the context's error slot and return code
int mrq_internal_fail(mrq_ctx* ctx, int code, const char* fmt, ...);
// Bytes the context's walk workspace may take from now on (a launch works in smaller segments and waves within
// them; a floor of 256 walkers and one determinant per wave remains).  A workspace above that is given back.
int mrq_internal_work_limit(mrq_ctx* ctx, long long bytes);
// Bytes of the floor for a system (0 where its sizes are out of range); that of a batch is below the sum over its systems
long long mrq_internal_work_floor(int n_core, int n_act, int n_virt, int n_alpha, int n_beta, long long n_ref);
// the context's host-wait (deadline-aware) synchronisation
int mrq_internal_sync(mrq_ctx* ctx);

#endif
