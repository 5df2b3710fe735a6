// The x + influence pass on the register engines, FP32.
#include "fft_xy.cuh"

namespace pppm {

typedef float T;
typedef Cx<T>::t C;

template <int L>
static cudaError_t run_x(cudaStream_t s, const Geo& g, const LineBlocks& lb, const C* tw, const T* G, T beta,
                         T e_scale, T c_field, C* S, C* Bx, T* partial) {
    auto kern = k_fft_x_reg<T, L>;
    constexpr size_t smem = x_smem<T, L>();
    const cudaError_t e = allow_smem(kern, smem);
    if (e != cudaSuccess) return e;
    return launch_k(kern, dim3(lb.nblk), dim3(FacS<L>::NT), smem, s, g, lb, tw, G, beta, e_scale, c_field, S, Bx,
                    partial);
}

template <>
cudaError_t reg_x_influence<T>(cudaStream_t s, const Geo& g, const LineBlocks& lb, const C* tw, const T* G,
                               double beta, double e_scale, double c_field, C* S, C* Bx, T* partial) {
    switch (g.N[0]) {
#define PPPM_LEN(L) \
    case L: return run_x<L>(s, g, lb, tw, G, (T)beta, (T)e_scale, (T)c_field, S, Bx, partial);
        PPPM_REG_LENGTHS(PPPM_LEN)
#undef PPPM_LEN
    }
    return cudaErrorNotSupported;
}

int reg_resident_x(T, int L) {
    switch (L) {
#define PPPM_LEN(LL) \
    case LL: return resident_blocks(k_fft_x_reg<T, LL>, FacS<LL>::NT, x_smem<T, LL>());
        PPPM_REG_LENGTHS(PPPM_LEN)
#undef PPPM_LEN
    }
    return 0;
}

}  // namespace pppm
