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
// Thread j of a line at `line`, its elements es apart; sm is the line's column
// of an exchange buffer (one barrier).
template <typename R, int L, int SIGN>
__device__ __forceinline__ void line_body(bool on, int j, typename CT<R>::C* sm,
                                          const typename CT<R>::C* __restrict__ tw,
                                          typename CT<R>::C* __restrict__ line, int64_t es) {
    typedef LineEngine<R, L> E;
    typedef typename CT<R>::C C;
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

// axis 1: lines along y (outer index x); axis 0: lines along x (outer index y)
template <typename R, int L, int SIGN>
__global__ void __launch_bounds__(FacS<L>::NT, pass_blocks<R, FacS<L>::NT>(40 + 5 * FacS<L>::A / 2))
k_fft_lines(Geo g, int axis, LineBlocks lb, const typename CT<R>::C* __restrict__ tw,
            typename CT<R>::C* __restrict__ data) {
    pdl_enter();
    typedef typename CT<R>::C C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int Hz = g.Hz;
    const int64_t es = axis == 1 ? (int64_t)Hz : (int64_t)g.N[1] * Hz;  // along the line
    const int64_t os = axis == 1 ? (int64_t)g.N[1] * Hz : (int64_t)Hz;  // between outer rows
    const int64_t nlines = (int64_t)(axis == 1 ? g.N[0] : g.N[1]) * Hz;
    const int64_t f = (int64_t)blockIdx.x * lb.B + (threadIdx.x & 15);
    const bool on = (int)(threadIdx.x & 15) < lb.B && f < nlines;
    line_body<R, L, SIGN>(on, threadIdx.x >> 4, reinterpret_cast<C*>(smem_raw) + (threadIdx.x & 15), tw,
                          data + (f / Hz) * os + f % Hz, es);
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
// end, by one block of at least 32 threads.  The sums are read past the L1: in
// a batch other blocks of the same launch wrote them (the caller has ordered
// their stores before this).
template <typename R>
__device__ __forceinline__ void finish_energy(const R* partial, int nblk, double prefactor,
                                              double* __restrict__ energy, double* __restrict__ virial) {
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    if ((int)(threadIdx.x >> 5) >= nw) return;  // a last warp that is not whole
    for (int q = threadIdx.x >> 5; q < 7; q += nw) {
        R h = R(0), lo = R(0);
        for (int b = lane; b < nblk; b += 32)
            two_sum_pair(h, lo, __ldcg(&partial[(int64_t)b * 14 + 2 * q]), __ldcg(&partial[(int64_t)b * 14 + 2 * q + 1]));
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
// one line's constants
template <typename R>
struct XLine {
    R kx, ky, kz;   // wavevector a step of the x index; the line's own y and z components
    R inv4b2;       // 1 / (4 beta^2)
    R e_scale, c_field;
    bool plane1;    // kz = 0 or Nz / 2: the mode stands for itself alone
    bool nyq_y;     // y is the Nyquist index of an even axis
};

template <typename R>
__device__ __forceinline__ XLine<R> x_line(const Geo& g, int y, int kz, R beta, R e_scale, R c_field) {
    XLine<R> m;
    m.kx = kfac<R>(g, 0);
    m.ky = kfac<R>(g, 1) * (y <= g.N[1] / 2 ? y : y - g.N[1]);
    m.kz = kfac<R>(g, 2) * kz;
    m.inv4b2 = R(1) / (R(4) * beta * beta);
    m.e_scale = e_scale;
    m.c_field = c_field;
    m.plane1 = kz == 0 || (g.N[2] % 2 == 0 && kz == g.N[2] / 2);
    m.nyq_y = g.N[1] % 2 == 0 && y == g.N[1] / 2;
    return m;
}

// Thread j of a line: S, Bx and G point at the line's first element, es apart;
// s0 and s1 are the line's columns of two exchange buffers; term gets the
// thread's energy and virial sums.  Every thread of the block calls it (three
// barriers; the buffers may be reused after one more).
template <typename R, int L>
__device__ __forceinline__ void x_body(bool on, int j, typename CT<R>::C* s0, typename CT<R>::C* s1,
                                       const typename CT<R>::C* __restrict__ tw, const R* __restrict__ G,
                                       typename CT<R>::C* __restrict__ S, typename CT<R>::C* __restrict__ Bx,
                                       int64_t es, const XLine<R>& m, R (&term)[7]) {
    typedef LineEngine<R, L> E;
    typedef typename CT<R>::C C;
    constexpr int A = E::A, B = E::B, T = E::T, G2 = E::G2;
    R gk[G2][B];
    if (on) {
        if (j < B) {
            C v[A];
#pragma unroll
            for (int n = 0; n < A; ++n) v[n] = S[(B * n + j) * es];
            E::template first<-1>(v, j, s0, tw);
        }
#pragma unroll
        for (int q = 0; q < G2; ++q)
#pragma unroll
            for (int k = 0; k < B; ++k) gk[q][k] = __ldg(&G[(j + T * q + A * k) * es]);
    }
    __syncthreads();
    C P[G2][B];
    R a_t = R(0), a_u = R(0), a_x = R(0), a_n = R(0), a_xx = R(0);
    if (on) {
        const R kyz = m.ky * m.ky + m.kz * m.kz;
#pragma unroll
        for (int q = 0; q < G2; ++q) E::template second<-1>(P[q], j + T * q, s0);
#pragma unroll
        for (int q = 0; q < G2; ++q) {
            C w[B];
#pragma unroll
            for (int k = 0; k < B; ++k) {
                const int i = j + T * q + A * k;
                const bool nyq = L % 2 == 0 && i == L / 2;
                const R kx = m.kx * (i <= L / 2 ? i : i - L);
                const C v = P[q][k];
                const R k2 = kx * kx + kyz;
                const R t = gk[q][k] * (v.x * v.x + v.y * v.y);
                const R u = t * ((k2 > R(0) ? recip(k2) : R(0)) + m.inv4b2);
                const R ux = u * kx;
                a_t += t;
                a_u += u;
                a_x += nyq ? R(0) : ux;
                a_n += nyq ? ux : R(0);
                a_xx += ux * kx;
                P[q][k] = cscale(v, gk[q][k] * m.c_field);
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
            for (int n = 0; n < A; ++n) Bx[(B * n + j) * es] = v[n];
        }
    }
    __syncthreads();
    if (on && j < B) {
        C v[A];
        E::template back_second<1>(v, j, s0);
#pragma unroll
        for (int n = 0; n < A; ++n) S[(B * n + j) * es] = v[n];
    }
    const R e1 = on ? (m.plane1 ? m.e_scale : R(2) * m.e_scale) : R(0), e2 = R(2) * e1;
    const R sxy = m.plane1 ? a_x + a_n : (m.nyq_y ? a_n : a_x);
    const R sxz = m.plane1 ? a_x + a_n : a_x;
    const R syz = (m.plane1 || !m.nyq_y) ? a_u : R(0);
    term[0] = e1 * a_t;
    term[1] = e1 * a_t - e2 * a_xx;
    term[2] = e1 * a_t - e2 * m.ky * m.ky * a_u;
    term[3] = e1 * a_t - e2 * m.kz * m.kz * a_u;
    term[4] = -e2 * m.ky * sxy;
    term[5] = -e2 * m.kz * sxz;
    term[6] = -e2 * m.ky * m.kz * syz;
}

// The block's sum of each term over its NT threads with compensated pairs, by
// its whole warps, to out[2 q], out[2 q + 1].  red: 7 NT values of shared
// memory that no thread uses any more.
template <typename R, int NT>
__device__ __forceinline__ void block_terms(const R (&term)[7], R* red, R* __restrict__ out) {
#pragma unroll
    for (int q = 0; q < 7; ++q) red[q * NT + threadIdx.x] = term[q];
    __syncthreads();
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31;
    if ((int)(threadIdx.x >> 5) >= NW) return;  // a last warp that is not whole
    for (int q = threadIdx.x >> 5; q < 7; q += NW) {
        R h = R(0), lo = R(0);
        for (int i = lane; i < NT; i += 32) two_sum_pair(h, lo, red[q * NT + i], R(0));
        for (int off = 16; off > 0; off >>= 1) {
            const R h2 = __shfl_down_sync(0xffffffffu, h, off);
            const R l2 = __shfl_down_sync(0xffffffffu, lo, off);
            two_sum_pair(h, lo, h2, l2);
        }
        if (lane == 0) {
            out[2 * q] = h;
            out[2 * q + 1] = lo;
        }
    }
}

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
    typedef typename CT<R>::C C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int64_t es = (int64_t)g.N[1] * g.Hz;
    const int l = threadIdx.x & 15, j = threadIdx.x >> 4;
    const int64_t f = (int64_t)blockIdx.x * lb.B + l;
    const bool on = l < lb.B && f < es;
    C* s0 = reinterpret_cast<C*>(smem_raw) + l;
    const int y = (int)(f / g.Hz), kz = (int)(f - (int64_t)y * g.Hz);
    R term[7];
    x_body<R, L>(on, j, s0, s0 + L * 16, tw, G + f, S + f, Bx + f, es, x_line<R>(g, y, kz, beta, e_scale, c_field),
                 term);
    __syncthreads();
    block_terms<R, FacS<L>::NT>(term, reinterpret_cast<R*>(smem_raw), partial + (int64_t)blockIdx.x * 14);
}

// ------------------------------------------------------------------ y inverse, three outputs
// C = IFFT_y(A), D = IFFT_y(-i ky' A), Ex' = IFFT_y(Bx); C overwrites A, Ex'
// overwrites Bx.  Block 0 sums the x pass's energy partials, the others take
// lb.B lines each.
//
// Thread j of a line: A, Bx and D point at the line's first element, es apart;
// s0 and s1 as in x_body (three barriers).
template <typename R, int L>
__device__ __forceinline__ void y_inv3_body(bool on, int j, typename CT<R>::C* s0, typename CT<R>::C* s1,
                                            const typename CT<R>::C* __restrict__ tw, R kfac_y,
                                            typename CT<R>::C* __restrict__ Am, typename CT<R>::C* __restrict__ Bx,
                                            typename CT<R>::C* __restrict__ D, int64_t es) {
    typedef LineEngine<R, L> E;
    typedef typename CT<R>::C C;
    constexpr int A = E::A, B = E::B, T = E::T, G2 = E::G2;
    C va[A];
    auto store = [&](C* __restrict__ out, const C* sm) {
#pragma unroll
        for (int q = 0; q < G2; ++q) {
            C u[B];
            E::template second<1>(u, j + T * q, sm);
#pragma unroll
            for (int k = 0; k < B; ++k) out[(j + T * q + A * k) * es] = u[k];
        }
    };
    if (on && j < B) {
        C v[A];
#pragma unroll
        for (int n = 0; n < A; ++n) v[n] = Bx[(B * n + j) * es];
#pragma unroll
        for (int n = 0; n < A; ++n) va[n] = Am[(B * n + j) * es];
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
                const R kyd = (L % 2 == 0 && m == L / 2) ? R(0) : kfac_y * (m <= L / 2 ? m : m - L);
                va[n] = CT<R>::mk(kyd * va[n].y, -kyd * va[n].x);
            }
            E::template first<1>(va, j, s0, tw);
        }
        store(Am, s1);
    }
    __syncthreads();
    if (on) store(D, s0);
}

template <typename R, int L>
__global__ void __launch_bounds__(FacS<L>::NT, pass_blocks<R, FacS<L>::NT>(56 + 4 * FacS<L>::A))
k_fft_y_inv3_reg(Geo g, LineBlocks lb, const typename CT<R>::C* __restrict__ tw, typename CT<R>::C* __restrict__ Am,
                 typename CT<R>::C* __restrict__ Bx, typename CT<R>::C* __restrict__ D, const R* __restrict__ partial,
                 int npart, double prefactor, double* __restrict__ energy, double* __restrict__ virial) {
    pdl_enter();
    typedef typename CT<R>::C C;
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
    y_inv3_body<R, L>(on, j, s0, s0 + L * 16, tw, kfac<R>(g, 1), Am + off, Bx + off, D + off, Hz);
}

}  // namespace pppm
