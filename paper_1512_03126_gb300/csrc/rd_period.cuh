// Constants of one operator-splitting period (Algorithm 1 of arXiv:1512.03126,
// Step 2 and Step 3), shared by the kernels.
#pragma once
#include "rd_device.cuh"
#include "rd_internal.h"

namespace rdk {

constexpr int kEventCap = 1 << 22;   // SSA events per tet and period
// Below this N* the diffusion draw is one uniform per molecule (the paper's
// per-molecule form, Sec. II.B); at or above it, Binomial + conditional
// binomials in double precision.
constexpr int64_t kMoleculeCut = 4096;
constexpr double kAvogadro = 6.02214076e23;

// Transfer probability over a period of length tau_k (Eq. 1 and the text
// after it): zeta = tau_k * D * G, at most 1.
__device__ __forceinline__ double zeta_of(double tau_k, double D, double Gt) {
    double z = tau_k * (D * Gt);
    return z > 1.0 ? 1.0 : z;
}

}  // namespace rdk
