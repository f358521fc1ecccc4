// The pack launch: companding, packing and the de-companding factors of a call.
#pragma once

#include "tdg_internal.h"

namespace tdg {

template <typename T>
struct PackArgs {
    PackOperand<T> A, B;      // op(A)[m][k] and op(B)[k][n] as (x, k), with block maxima
    T *outA, *outB;
    // leading dimension of the packed A by W (the asymmetric form's differs),
    // [0]: of its plain copy
    long long ldoA[kMaxW + 1], ldoB;
    T *pair;                  // nullable: [l][i][j] factors
    int L, nM, nK, nN;
    int target;               // the plan may have fallen back to the plain product
    int plain;                // plain copies whatever the plan says
    int plain_only;           // only the fallback's plain copies
    int directA, directB;     // the plain product reads this operand in place
    int skipA, skipB;         // operand kept from an earlier call
    int manual;
    double manual_cA, manual_cB;
    // set by the launcher: tiles of factors; CTAs that pack, and the index of the
    // one after them (targets only)
    int pair_tiles;
    unsigned int log_cta;
};

// One launch over both operands for whichever W the device plan holds (along k:
// the symmetric form and plain copies; asym: A along x, B unpacked).
template <typename T>
cudaError_t launch_pack(bool asym, const PackArgs<T> &a, DevPlan *plan, cudaStream_t st);

}  // namespace tdg
