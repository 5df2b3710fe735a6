// The strided passes (lines along x and y) on the register engines: see
// fft_reg.cuh for the transform and fft_kernels.cu for the passes' place in
// the solve.  Included by the translation units that instantiate them.
//
// A block holds up to 16 consecutive lines (lane tid % 16) of the flattened
// (outer, kz) index and T threads a line (tid / 16): a row of 16 lines is 128
// contiguous bytes in global memory and free of bank conflicts in shared
// memory, where point i of line l is at i 16 + l.
#pragma once

#include "fft_reg.cuh"

namespace pppm {

template <typename R, int L>
struct LineEngine : FacS<L> {
    typedef typename CT<R>::C C;
    using F = FacS<L>;
    static constexpr int A = F::A, B = F::B;
    static constexpr size_t kBytes = sizeof(C) * L * 16;  // one exchange buffer

    // stage 1 of butterfly n2 = j into shared memory (column of this line)
    template <int SIGN>
    static __device__ __forceinline__ void first(C (&v)[A], int j, C* sm, const C* __restrict__ tw) {
        dft<C, R, A, SIGN>(v);
        sm[j * 16] = v[0];
#pragma unroll
        for (int k = 1; k < A; ++k) sm[(k * B + j) * 16] = cmul(v[k], twiddle<R, SIGN>(tw, j * k));
    }
    // stage 2 of k1: v[k2] = X[k1 + A k2]
    template <int SIGN>
    static __device__ __forceinline__ void second(C (&v)[B], int k1, const C* sm) {
#pragma unroll
        for (int n = 0; n < B; ++n) v[n] = sm[(k1 * B + n) * 16];
        dft<C, R, B, SIGN>(v);
    }
    // the same backwards: stage 2 of k1 from v[k2] = X[k1 + A k2] ...
    template <int SIGN>
    static __device__ __forceinline__ void back_first(C (&v)[B], int k1, C* sm, const C* __restrict__ tw) {
        dft<C, R, B, SIGN>(v);
        sm[(k1 * B) * 16] = v[0];
#pragma unroll
        for (int n = 1; n < B; ++n) sm[(k1 * B + n) * 16] = cmul(v[n], twiddle<R, SIGN>(tw, k1 * n));
    }
    // ... and stage 1 of n2 = j: v[n1] = x[B n1 + j]
    template <int SIGN>
    static __device__ __forceinline__ void back_second(C (&v)[A], int j, const C* sm) {
#pragma unroll
        for (int k = 0; k < A; ++k) v[k] = sm[(k * B + j) * 16];
        dft<C, R, A, SIGN>(v);
    }
};

// ------------------------------------------------------------------ one transform in place
// axis 1: lines along y (outer index x); axis 0: lines along x (outer index y)
template <typename R, int L, int SIGN>
__global__ void __launch_bounds__(FacS<L>::NT, pass_blocks<R, FacS<L>::NT>(40 + 5 * FacS<L>::A / 2))
k_fft_lines(Geo g, int axis, LineBlocks lb, const typename CT<R>::C* __restrict__ tw,
            typename CT<R>::C* __restrict__ data) {
    pdl_enter();
    typedef LineEngine<R, L> E;
    typedef typename CT<R>::C C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int Hz = g.Hz;
    const int64_t es = axis == 1 ? (int64_t)Hz : (int64_t)g.N[1] * Hz;  // along the line
    const int64_t os = axis == 1 ? (int64_t)g.N[1] * Hz : (int64_t)Hz;  // between outer rows
    const int64_t nlines = (int64_t)(axis == 1 ? g.N[0] : g.N[1]) * Hz;
    const int64_t f = (int64_t)blockIdx.x * lb.B + (threadIdx.x & 15);
    const bool on = (int)(threadIdx.x & 15) < lb.B && f < nlines;
    const int j = threadIdx.x >> 4;
    C* line = data + (f / Hz) * os + f % Hz;
    C* sm = reinterpret_cast<C*>(smem_raw) + (threadIdx.x & 15);
    if (on && j < E::B) {
        C v[E::A];
#pragma unroll
        for (int n = 0; n < E::A; ++n) v[n] = line[(E::B * n + j) * es];
        E::template first<SIGN>(v, j, sm, tw);
    }
    __syncthreads();
    if (!on) return;
#pragma unroll
    for (int q = 0; q < E::G2; ++q) {
        const int k1 = j + E::T * q;
        C u[E::B];
        E::template second<SIGN>(u, k1, sm);
#pragma unroll
        for (int k = 0; k < E::B; ++k) line[(k1 + E::A * k) * es] = u[k];
    }
}

// ------------------------------------------------------------------ energy and virial partials
// (h, l) += (h2, l2) with the rounding error of h + h2 carried into l
template <typename R>
__device__ __forceinline__ void two_sum_pair(R& h, R& l, R h2, R l2) {
    R s = h + h2;
    R bp = s - h;
    R err = (h - (s - bp)) + (h2 - bp);
    h = s;
    l = l + l2 + err;
}

// Sums the x pass's per-block partials (14 values a block: 7 (hi, lo) pairs)
// in a fixed order, TwoSum in the mesh precision and hi + lo in FP64 at the
// end, by one block of at least 32 threads.
template <typename R>
__device__ __forceinline__ void finish_energy(const R* __restrict__ partial, int nblk, double prefactor,
                                              double* __restrict__ energy, double* __restrict__ virial) {
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    if ((int)(threadIdx.x >> 5) >= nw) return;  // a last warp that is not whole
    for (int q = threadIdx.x >> 5; q < 7; q += nw) {
        R h = R(0), lo = R(0);
        for (int b = lane; b < nblk; b += 32)
            two_sum_pair(h, lo, partial[(int64_t)b * 14 + 2 * q], partial[(int64_t)b * 14 + 2 * q + 1]);
        for (int off = 16; off > 0; off >>= 1) {
            const R h2 = __shfl_down_sync(0xffffffffu, h, off);
            const R l2 = __shfl_down_sync(0xffffffffu, lo, off);
            two_sum_pair(h, lo, h2, l2);
        }
        if (lane == 0) {
            const double sum = ((double)h + (double)lo) * prefactor;
            if (q == 0) energy[0] = sum;
            else virial[q - 1] = sum;
        }
    }
}

// 1 / k^2 for the virial: in FP32 the hardware reciprocal (the coefficient
// enters sums that are accurate to ~1e-7 anyway), in FP64 exact
__device__ __forceinline__ float recip(float a) { return __fdividef(1.f, a); }
__device__ __forceinline__ double recip(double a) { return 1.0 / a; }

// ------------------------------------------------------------------ x + influence
// Per block: 16 lines along x, numbered y Hz + kz.  The forward transform
// leaves a thread's modes k1 + A k2 in its registers; there they are
// multiplied by the influence function (P = G rho_hat / (N h^3)) and give
// their energy and virial terms, and the inverse transforms of -i kx' P and
// of P start from the same registers.
//
// On one line ky and kz are fixed, so the seven sums are formed per line from
// five: with t = G |rho_hat|^2 and u = t (1 / k^2 + 1 / (4 beta^2)),
//   sum t, sum u, sum u kx (without the Nyquist index of an even axis), that
//   index's own u kx, and sum u kx^2
// (e = w e_scale t and e c = 2 w e_scale u; the terms are e (delta_ab - c k_a
// k_b)).  Half-spectrum weights and the Nyquist rule of the off-diagonal terms
// are those described at the pass in fft_kernels.cu.
template <typename R, int L>
constexpr size_t x_smem() {
    typedef LineEngine<R, L> E;
    return 2 * E::kBytes > 7 * sizeof(R) * E::NT ? 2 * E::kBytes : 7 * sizeof(R) * E::NT;
}

template <typename R, int L>
__global__ void __launch_bounds__(FacS<L>::NT,
                                  pass_blocks<R, FacS<L>::NT>(56 + 2 * FacS<L>::G2 * FacS<L>::B + 2 * FacS<L>::A))
k_fft_x_reg(Geo g, LineBlocks lb, const typename CT<R>::C* __restrict__ tw, const R* __restrict__ G, R beta, R e_scale,
            R c_field, typename CT<R>::C* __restrict__ S, typename CT<R>::C* __restrict__ Bx,
            R* __restrict__ partial) {
    pdl_enter();
    typedef LineEngine<R, L> E;
    typedef typename CT<R>::C C;
    constexpr int A = E::A, B = E::B, T = E::T, G2 = E::G2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int Ny = g.N[1], Nz = g.N[2], Hz = g.Hz;
    const int64_t es = (int64_t)Ny * Hz;
    const int l = threadIdx.x & 15, j = threadIdx.x >> 4;
    const int64_t f = (int64_t)blockIdx.x * lb.B + l;
    const bool on = l < lb.B && f < es;
    C* s0 = reinterpret_cast<C*>(smem_raw) + l;
    C* s1 = s0 + L * 16;
    R gk[G2][B];
    if (on) {
        if (j < B) {
            C v[A];
#pragma unroll
            for (int n = 0; n < A; ++n) v[n] = S[(B * n + j) * es + f];
            E::template first<-1>(v, j, s0, tw);
        }
#pragma unroll
        for (int q = 0; q < G2; ++q)
#pragma unroll
            for (int k = 0; k < B; ++k) gk[q][k] = __ldg(&G[(j + T * q + A * k) * es + f]);
    }
    __syncthreads();
    C P[G2][B];
    R a_t = R(0), a_u = R(0), a_x = R(0), a_n = R(0), a_xx = R(0);
    const int y = (int)(f / Hz), kz = (int)(f - (int64_t)y * Hz);
    const R ky = kfac<R>(g, 1) * (y <= Ny / 2 ? y : y - Ny), kzv = kfac<R>(g, 2) * kz;
    if (on) {
        const R kyz = ky * ky + kzv * kzv;
        const R inv4b2 = R(1) / (R(4) * beta * beta);
#pragma unroll
        for (int q = 0; q < G2; ++q) E::template second<-1>(P[q], j + T * q, s0);
#pragma unroll
        for (int q = 0; q < G2; ++q) {
            C w[B];
#pragma unroll
            for (int k = 0; k < B; ++k) {
                const int m = j + T * q + A * k;
                const bool nyq = L % 2 == 0 && m == L / 2;
                const R kx = kfac<R>(g, 0) * (m <= L / 2 ? m : m - L);
                const C v = P[q][k];
                const R k2 = kx * kx + kyz;
                const R t = gk[q][k] * (v.x * v.x + v.y * v.y);
                const R u = t * ((k2 > R(0) ? recip(k2) : R(0)) + inv4b2);
                const R ux = u * kx;
                a_t += t;
                a_u += u;
                a_x += nyq ? R(0) : ux;
                a_n += nyq ? ux : R(0);
                a_xx += ux * kx;
                P[q][k] = cscale(v, gk[q][k] * c_field);
                const R kxd = nyq ? R(0) : kx;
                w[k] = CT<R>::mk(kxd * P[q][k].y, -kxd * P[q][k].x);  // -i kx' P
            }
            E::template back_first<1>(w, j + T * q, s1, tw);
        }
    }
    __syncthreads();  // s0 has been read, s1 written
    if (on) {
#pragma unroll
        for (int q = 0; q < G2; ++q) E::template back_first<1>(P[q], j + T * q, s0, tw);
        if (j < B) {
            C v[A];
            E::template back_second<1>(v, j, s1);
#pragma unroll
            for (int n = 0; n < A; ++n) Bx[(B * n + j) * es + f] = v[n];
        }
    }
    __syncthreads();
    if (on && j < B) {
        C v[A];
        E::template back_second<1>(v, j, s0);
#pragma unroll
        for (int n = 0; n < A; ++n) S[(B * n + j) * es + f] = v[n];
    }
    __syncthreads();
    // this thread's seven terms, reduced over the block with compensated pairs
    R* red = reinterpret_cast<R*>(smem_raw);
    {
        const bool plane1 = (kz == 0) || (Nz % 2 == 0 && kz == Nz / 2);
        const bool nyq_y = Ny % 2 == 0 && y == Ny / 2;
        const R e1 = on ? (plane1 ? e_scale : R(2) * e_scale) : R(0), e2 = R(2) * e1;
        const R sxy = plane1 ? a_x + a_n : (nyq_y ? a_n : a_x);
        const R sxz = plane1 ? a_x + a_n : a_x;
        const R syz = (plane1 || !nyq_y) ? a_u : R(0);
        const R term[7] = {e1 * a_t,
                           e1 * a_t - e2 * a_xx,
                           e1 * a_t - e2 * ky * ky * a_u,
                           e1 * a_t - e2 * kzv * kzv * a_u,
                           -e2 * ky * sxy,
                           -e2 * kzv * sxz,
                           -e2 * ky * kzv * syz};
#pragma unroll
        for (int q = 0; q < 7; ++q) red[q * E::NT + threadIdx.x] = term[q];
    }
    __syncthreads();
    constexpr int NW = E::NT / 32;
    const int lane = threadIdx.x & 31;
    if ((int)(threadIdx.x >> 5) >= NW) return;  // a last warp that is not whole
    for (int q = threadIdx.x >> 5; q < 7; q += NW) {
        R h = R(0), lo = R(0);
        for (int i = lane; i < E::NT; i += 32) two_sum_pair(h, lo, red[q * E::NT + i], R(0));
        for (int off = 16; off > 0; off >>= 1) {
            const R h2 = __shfl_down_sync(0xffffffffu, h, off);
            const R l2 = __shfl_down_sync(0xffffffffu, lo, off);
            two_sum_pair(h, lo, h2, l2);
        }
        if (lane == 0) {
            partial[(int64_t)blockIdx.x * 14 + 2 * q] = h;
            partial[(int64_t)blockIdx.x * 14 + 2 * q + 1] = lo;
        }
    }
}

// ------------------------------------------------------------------ y inverse, three outputs
// C = IFFT_y(A), D = IFFT_y(-i ky' A), Ex' = IFFT_y(Bx); C overwrites A, Ex'
// overwrites Bx.  Block 0 sums the x pass's energy partials, the others take
// lb.B lines each.
template <typename R, int L>
__global__ void __launch_bounds__(FacS<L>::NT, pass_blocks<R, FacS<L>::NT>(56 + 4 * FacS<L>::A))
k_fft_y_inv3_reg(Geo g, LineBlocks lb, const typename CT<R>::C* __restrict__ tw, typename CT<R>::C* __restrict__ Am,
                 typename CT<R>::C* __restrict__ Bx, typename CT<R>::C* __restrict__ D, const R* __restrict__ partial,
                 int npart, double prefactor, double* __restrict__ energy, double* __restrict__ virial) {
    pdl_enter();
    typedef LineEngine<R, L> E;
    typedef typename CT<R>::C C;
    constexpr int A = E::A, B = E::B, T = E::T, G2 = E::G2;
    if (blockIdx.x == 0) {
        finish_energy(partial, npart, prefactor, energy, virial);
        return;
    }
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int Hz = g.Hz;
    const int l = threadIdx.x & 15, j = threadIdx.x >> 4;
    const int64_t f = (int64_t)(blockIdx.x - 1) * lb.B + l;
    const bool on = l < lb.B && f < (int64_t)g.N[0] * Hz;
    const int64_t off = (f / Hz) * ((int64_t)L * Hz) + f % Hz;
    C* s0 = reinterpret_cast<C*>(smem_raw) + l;
    C* s1 = s0 + L * 16;
    C va[A];
    auto store = [&](C* __restrict__ out, const C* sm) {
#pragma unroll
        for (int q = 0; q < G2; ++q) {
            C u[B];
            E::template second<1>(u, j + T * q, sm);
#pragma unroll
            for (int k = 0; k < B; ++k) out[off + (int64_t)(j + T * q + A * k) * Hz] = u[k];
        }
    };
    if (on && j < B) {
        C v[A];
#pragma unroll
        for (int n = 0; n < A; ++n) v[n] = Bx[off + (int64_t)(B * n + j) * Hz];
#pragma unroll
        for (int n = 0; n < A; ++n) va[n] = Am[off + (int64_t)(B * n + j) * Hz];
        E::template first<1>(v, j, s0, tw);
    }
    __syncthreads();
    if (on) {
        if (j < B) {
            C v[A];
#pragma unroll
            for (int n = 0; n < A; ++n) v[n] = va[n];
            E::template first<1>(v, j, s1, tw);
        }
        store(Bx, s0);
    }
    __syncthreads();
    if (on) {
        if (j < B) {
#pragma unroll
            for (int n = 0; n < A; ++n) {
                const int m = B * n + j;
                const R kyd = (L % 2 == 0 && m == L / 2) ? R(0) : kfac<R>(g, 1) * (m <= L / 2 ? m : m - L);
                va[n] = CT<R>::mk(kyd * va[n].y, -kyd * va[n].x);
            }
            E::template first<1>(va, j, s0, tw);
        }
        store(Am, s1);
    }
    __syncthreads();
    if (on) store(D, s0);
}

}  // namespace pppm
