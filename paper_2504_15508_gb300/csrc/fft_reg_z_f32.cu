// The z passes on the register engines, FP32.
#include "fft_z.cuh"

namespace pppm {

typedef float T;
typedef Cx<T>::t C;

// pairs a block: at most `most`, fewer when that would leave SMs without a
// block, but no less than a warp's threads
template <int L>
static int pairs_per_block(int pairs, int threads, int most) {
    const int least = (32 + threads - 1) / threads, nsm = device_sms();
    int np = (pairs + nsm - 1) / nsm;
    np = np < least ? least : np;
    return np > most ? most : np;
}

template <int L>
static cudaError_t run_r2c(cudaStream_t s, const Geo& g, const C* tw, const T* in, C* out, const PatchSrc<T>& ps) {
    typedef FacF<T, L> F;
    const int rows = g.N[0] * g.N[1], pairs = (rows + 1) / 2, np = pairs_per_block<L>(pairs, F::T, F::NPMAX);
    // two sets of threads fold a pair's rows while one set does not fill the
    // GPU (about 320 threads an SM): 90^3 22.0 -> 16.8 us, 64^3 12.2 -> 11.4,
    // but 128^3 16.3 -> 17.7, 160^3 25.8 -> 28.8
    const bool split = ps.patch && (int64_t)pairs * F::T < device_sms() * 320;
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
        const int np = pairs_per_block<L>(pairs, F::T, F::NPMAX);
        const size_t smem = sizeof(C) * F::PITCH * np;
        auto kern = k_fft_z_c2r_plain<T, L>;
        const cudaError_t e = allow_smem(kern, smem);
        if (e != cudaSuccess) return e;
        return launch_k(kern, dim3((pairs + np - 1) / np, zo.nf), dim3(np * F::T), smem, s, g, tw, zo, rows);
    }
    const int np = pairs_per_block<L>(pairs, zo.nf * F::T, FacC2R<T, L>::NT / (zo.nf * F::T));
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
        PPPM_REG_LENGTHS(PPPM_LEN)
#undef PPPM_LEN
    }
    return cudaErrorNotSupported;
}

template <>
cudaError_t reg_z_c2r<T>(cudaStream_t s, const Geo& g, const C* tw, const ZOut& zo) {
    switch (g.N[2]) {
#define PPPM_LEN(L) \
    case L: return run_c2r<L>(s, g, tw, zo);
        PPPM_REG_LENGTHS(PPPM_LEN)
#undef PPPM_LEN
    }
    return cudaErrorNotSupported;
}

}  // namespace pppm
