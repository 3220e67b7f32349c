// FP64 plans: the Tucker sums of a step as phases of grouped mode products.
// Internal interface (step64.cu).
#pragma once

#include <map>
#include <utility>
#include <vector>

#include "mm64.h"

namespace ds {

// plain: out (+)= sum_i eta_i T(X, {P[c][slot][i][mu]}), or its real part for
// the complex scheme; transposed: with the transposed matrices, times the
// slot's weight (the adjoint operator); tangent: the derivative of plain with
// respect to a scaling of component c's matrices.
enum class SumKind { plain, transposed, tangent };
struct SumOp {
    int c, slot;
    const double *X;
    double *out;
    bool accumulate = false;
};
// sums that run in one call
struct SumGroup {
    SumKind kind;
    std::vector<int> slots;   // each for both components
};

struct Sums64 {
    const ds_phi_set *set = nullptr;
    int64_t N = 0;
    mm::Context ctx;          // scratch for the tensors' digit images
    double *z = nullptr;      // intermediates between modes, z_tensors x N (the caller's memory)
    int64_t z_tensors = 0;
    uint8_t *mats = nullptr;  // digit images of the matrices, by view
    std::map<std::vector<long long>, mm::Image> images;
};

// intermediates of one sum (its z tensors); one term's share is 1 / k of it
int sum_tensors(const ds_phi_set *s, SumKind kind);
// Allocates scratch and cuts the matrices of `groups` into digits (on st, which
// it waits for).  Where memory is short the sums still run: matrices cut per
// call, or products on the FP64 pipe.
void sums_create(Sums64 &e, const ds_phi_set *s, int64_t N, const std::vector<SumGroup> &groups, double *z,
                 int64_t z_tensors, cudaStream_t st);
void sums_destroy(Sums64 &e);
// Runs independent sums of one kind; returns the number of launches.
int run_sums(const Sums64 &e, SumKind kind, const SumOp *ops, int count, Prof *prof, cudaStream_t st);
// One term's Tucker operator with its derivative matrix in mode `md`, of component c:
// out = T(X, P with P_md -> dP_md).  Two intermediates; returns the number of launches.
int run_partial(const Sums64 &e, int c, int slot, int term, int md, const double *X, double *out, Prof *prof, cudaStream_t st);
// Y_c = sum_mu X_c x_mu A_{c,mu} (transposed: A^T) for both components
int run_kronsum(const Sums64 &e, const double *X, double *Y, int transpose, Prof *prof, cudaStream_t st);

}  // namespace ds
