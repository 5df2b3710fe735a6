// The y passes (and the plain x transforms) on the register engines, FP32.
#include "fft_xy.cuh"

namespace pppm {

typedef float T;
typedef Cx<T>::t C;

template <int L>
static cudaError_t run_lines(cudaStream_t s, const Geo& g, int axis, int sign, const LineBlocks& lb, const C* tw,
                             C* data) {
    auto kern = sign < 0 ? k_fft_lines<T, L, -1> : k_fft_lines<T, L, 1>;
    constexpr size_t smem = LineEngine<T, L>::kBytes;
    const cudaError_t e = allow_smem(kern, smem);
    if (e != cudaSuccess) return e;
    return launch_k(kern, dim3(lb.nblk), dim3(FacS<L>::NT), smem, s, g, axis, lb, tw, data);
}

template <int L>
static cudaError_t run_inv3(cudaStream_t s, const Geo& g, const LineBlocks& lb, const C* tw, C* A, C* Bx, C* D,
                            const T* partial, int npart, double prefactor, double* energy, double* virial) {
    auto kern = k_fft_y_inv3_reg<T, L>;
    constexpr size_t smem = 2 * LineEngine<T, L>::kBytes;
    const cudaError_t e = allow_smem(kern, smem);
    if (e != cudaSuccess) return e;
    return launch_k(kern, dim3(lb.nblk + 1), dim3(FacS<L>::NT), smem, s, g, lb, tw, A, Bx, D, partial, npart,
                    prefactor, energy, virial);
}

template <>
cudaError_t reg_lines<T>(cudaStream_t s, const Geo& g, int axis, int sign, const LineBlocks& lb, const C* tw,
                         C* data) {
    switch (g.N[axis]) {
#define PPPM_LEN(L) \
    case L: return run_lines<L>(s, g, axis, sign, lb, tw, data);
        PPPM_REG_LENGTHS(PPPM_LEN)
#undef PPPM_LEN
    }
    return cudaErrorNotSupported;
}

template <>
cudaError_t reg_y_inverse3<T>(cudaStream_t s, const Geo& g, const LineBlocks& lb, const C* tw, C* A, C* Bx, C* D,
                              const T* partial, int npart, double prefactor, double* energy, double* virial) {
    switch (g.N[1]) {
#define PPPM_LEN(L) \
    case L: return run_inv3<L>(s, g, lb, tw, A, Bx, D, partial, npart, prefactor, energy, virial);
        PPPM_REG_LENGTHS(PPPM_LEN)
#undef PPPM_LEN
    }
    return cudaErrorNotSupported;
}

int reg_resident_x(T, int L);

template <>
int reg_resident<T>(int pass, int L) {
    if (pass == LB_X_INFLUENCE) return reg_resident_x(T(0), L);
    switch (L) {
#define PPPM_LEN(LL)                                                                                             \
    case LL:                                                                                                     \
        return pass == LB_Y_INVERSE3                                                                             \
                   ? resident_blocks(k_fft_y_inv3_reg<T, LL>, FacS<LL>::NT, 2 * LineEngine<T, LL>::kBytes)       \
                   : resident_blocks(k_fft_lines<T, LL, -1>, FacS<LL>::NT, LineEngine<T, LL>::kBytes);
        PPPM_REG_LENGTHS(PPPM_LEN)
#undef PPPM_LEN
    }
    return 0;
}

}  // namespace pppm
