// The z passes on the register engines, FP64.
#include <algorithm>
#include <cstdint>

#include "fft_z.cuh"

namespace pppm {

typedef double T;
typedef Cx<T>::t C;

// Pairs a block, of `threads` threads each, at most `most`.  The arithmetic of the
// busiest SM is what these passes wait for, so of the blocks of at least `warps`
// warps those are taken that give it the fewest (the larger of equal ones); a mesh
// too small for them gives every SM a block, of no less than a warp's threads.
// With as many pairs as fit, 176 blocks on 152 SMs take the time of 304:
// z inverse 60^3 42.9 -> 29.9 us, 45 x 60 x 75 49.1 -> 34.8, 100^3 189 -> 172; z
// forward 80^3 42.9 -> 34.8, 64 x 80 x 128 55.1 -> 43.1, with the seam rule of
// fold_row 75^3 62.5 -> 45.9.
static int pairs_per_block(int pairs, int threads, int most, int warps) {
    const int nsm = device_sms(), least = (32 * warps - 31 + threads - 1) / threads;
    const int even = std::max((pairs + nsm - 1) / nsm, (32 + threads - 1) / threads);
    if (even < least || least > most) return std::min(even, most);
    int best = most;
    int64_t busy = INT64_MAX;
    for (int np = most; np >= least; --np) {
        const int blocks = (pairs + np - 1) / np;
        const int64_t w = (int64_t)((blocks + nsm - 1) / nsm) * ((np * threads + 31) / 32);
        if (w < busy) {
            busy = w;
            best = np;
        }
    }
    return best;
}

template <int L>
static cudaError_t run_r2c(cudaStream_t s, const Geo& g, const C* tw, const T* in, C* out, const PatchSrc<T>& ps) {
    typedef FacF<T, L> F;
    const int rows = g.N[0] * g.N[1], pairs = (rows + 1) / 2;
    // two sets of threads fold a pair's rows while one set does not fill the
    // GPU (about 320 threads an SM): 32^3 18.3 -> 14.2 us, 64^3 30.8 -> 25.0,
    // 90^3 95.6 -> 91.1; from 96^3 on no difference
    const bool split = ps.patch && (int64_t)pairs * F::T < device_sms() * 320;
    const int np = pairs_per_block(pairs, (split ? 2 : 1) * F::T, F::NPMAX, 4);
    const size_t smem = sizeof(C) * F::PITCH * np;
    auto kern = split ? k_fft_z_r2c_reg<T, L, true> : k_fft_z_r2c_reg<T, L, false>;
    const cudaError_t e = allow_smem(kern, smem);
    if (e != cudaSuccess) return e;
    return launch_k(kern, dim3((pairs + np - 1) / np), dim3((split ? 2 : 1) * np * F::T), smem, s, g, tw, in, out, rows, ps);
}

template <int L>
static cudaError_t run_c2r(cudaStream_t s, const Geo& g, const C* tw, const ZOut& zo) {
    typedef FacI<T, L> F;
    const int rows = g.N[0] * g.N[1], pairs = (rows + 1) / 2;
    if (!zo.fl.padded) {
        const int np = pairs_per_block(pairs, F::T, F::NPMAX, 3);
        const size_t smem = sizeof(C) * F::PITCH * np;
        auto kern = k_fft_z_c2r_plain<T, L>;
        const cudaError_t e = allow_smem(kern, smem);
        if (e != cudaSuccess) return e;
        return launch_k(kern, dim3((pairs + np - 1) / np, zo.nf), dim3(np * F::T), smem, s, g, tw, zo, rows);
    }
    const int np = pairs_per_block(pairs, zo.nf * F::T, FacC2R<T, L>::NT / (zo.nf * F::T), 3);
    const size_t smem = c2r_pair_bytes<T, L>(zo.nf) * np;
    auto kern = k_fft_z_c2r_reg<T, L>;
    const cudaError_t e = allow_smem(kern, smem);
    if (e != cudaSuccess) return e;
    return launch_k(kern, dim3((pairs + np - 1) / np), dim3(np * zo.nf * F::T), smem, s, g, tw, zo, rows);
}

template <>
cudaError_t reg_z_r2c<T>(cudaStream_t s, const Geo& g, const C* tw, const T* in, C* out, const PatchSrc<T>& ps) {
    switch (g.N[2]) {
#define PPPM_LEN(L) \
    case L: return run_r2c<L>(s, g, tw, in, out, ps);
        PPPM_REG_LENGTHS_F64(PPPM_LEN)
#undef PPPM_LEN
    }
    return cudaErrorNotSupported;
}

template <>
cudaError_t reg_z_c2r<T>(cudaStream_t s, const Geo& g, const C* tw, const ZOut& zo) {
    switch (g.N[2]) {
#define PPPM_LEN(L) \
    case L: return run_c2r<L>(s, g, tw, zo);
        PPPM_REG_LENGTHS_F64(PPPM_LEN)
#undef PPPM_LEN
    }
    return cudaErrorNotSupported;
}

}  // namespace pppm
