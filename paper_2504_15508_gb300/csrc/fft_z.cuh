// The z passes on the register engines: see fft_reg.cuh for the transform and
// fft_kernels.cu for the passes' place in the solve.  Included by the
// translation units that instantiate them.
//
// A line is two real rows as one complex row, or two real fields of one row.
// Its T threads are consecutive, so that a step of a transform touches T
// consecutive points; with the frequencies k1 and A - k1 in one thread of the
// spectral side, a mode and its Hermitian mirror are in the same registers:
// the two real rows are separated (forward) or joined (inverse) without
// another exchange, and each half-spectrum value is read or written once.
#pragma once

#include "fft_reg.cuh"

namespace pppm {

// a line's exchange in shared memory: points (k1, n2) at k1 (B + 1) + n2
template <typename R, int L, int CAP = kPairCap<R>>
struct PairEngine : FacZ<L, CAP> {
    typedef typename CT<R>::C C;
    using F = FacZ<L, CAP>;
    static constexpr int A = F::A, B = F::B, T = F::T, T2 = F::T2, G1 = F::G1;

    // the line's other threads have written what this one reads next (every
    // thread of the block that has not returned takes part)
    static __device__ __forceinline__ void sync() {
        if constexpr (F::kWarp) __syncwarp();
        else __syncthreads();
    }
    // space side, forward: the DFT over n1 of butterfly n2, twiddled
    static __device__ __forceinline__ void space_out(C (&v)[A], int n2, C* sm, const C* __restrict__ tw) {
        dft<C, R, A, -1>(v);
        sm[n2] = v[0];
#pragma unroll
        for (int k = 1; k < A; ++k) sm[k * (B + 1) + n2] = cmul(v[k], twiddle<R, -1>(tw, n2 * k));
    }
    // spectral side, forward: Z[k1 + A k2]
    static __device__ __forceinline__ void spec_in(C (&v)[B], int k1, const C* sm) {
#pragma unroll
        for (int n = 0; n < B; ++n) v[n] = sm[k1 * (B + 1) + n];
        dft<C, R, B, -1>(v);
    }
    // the same backwards
    static __device__ __forceinline__ void spec_out(C (&v)[B], int k1, C* sm, const C* __restrict__ tw) {
        dft<C, R, B, 1>(v);
        sm[k1 * (B + 1)] = v[0];
#pragma unroll
        for (int n = 1; n < B; ++n) sm[k1 * (B + 1) + n] = cmul(v[n], twiddle<R, 1>(tw, k1 * n));
    }
    static __device__ __forceinline__ void space_in(C (&v)[A], int n2, const C* sm) {
#pragma unroll
        for (int k = 0; k < A; ++k) v[k] = sm[k * (B + 1) + n2];
        dft<C, R, A, 1>(v);
    }
};

// second frequency of thread j of the spectral side: A - j, and A / 2 for
// thread 0 (none for an odd A)
template <int A>
__device__ __forceinline__ int pair_k1(int j) {
    return j > 0 ? A - j : A / 2;
}
template <int A>
__device__ __forceinline__ bool pair_on(int j) {
    return j > 0 ? 2 * j != A : A % 2 == 0;
}

// ------------------------------------------------------------------ z forward (R2C)
// Rows of the mesh, or of the spread's tile patches summed on the way (the
// fold): mesh index m of an axis is covered by at most four (tile, patch
// coordinate) pairs, two away from a ragged last tile, listed in a fixed order
// (ps.cov: x entries; ps.off: y and z entries as offsets into the patches).
//
// The fold's dependent rounds of loads are the pass's longest chain.  On a mesh
// too small to hide it behind other warps (SPLIT), a pair's two rows are
// folded by two sets of threads: the second half of the block takes the odd
// rows and hands them over through shared memory.
//
// Sum of the patches at the A points z = B n + n2 of row (x, y).  SEAM: indices
// with more than two covers lie where near_seam says, so that only those n look
// them up (75^3 FP64 76.9 -> 62.5 us, 225^3 FP32 116 -> 91); else anywhere.
template <typename R, int A, int B, bool SEAM>
__device__ __forceinline__ void fold_row(const Geo& g, const PatchSrc<R>& ps, int row, int n2, R (&v)[A]) {
    const int4* zoff = ps.off + ps.nmax + n2;  // this thread's points: zoff[B n]
    int2 oz[A];
#pragma unroll
    for (int n = 0; n < A; ++n) {
        oz[n] = __ldg(reinterpret_cast<const int2*>(&zoff[B * n]));
        v[n] = R(0);
    }
    const int x = row / g.N[1], y = row - x * g.N[1];
    const int4 oy = __ldg(&ps.off[y]);
#pragma unroll 1
    for (int a = 0; a < 4; ++a) {
        const int2 cx = __ldg(&ps.cov[4 * x + a]);
        if (cx.x < 0) break;
        const R* px = ps.patch + (int64_t)cx.x * ps.xstride + cx.y * (g.E[1] * g.Pz);
#pragma unroll 1
        for (int b = 0; b < 4; ++b) {
            const int ob = b == 0 ? oy.x : b == 1 ? oy.y : b == 2 ? oy.z : oy.w;
            if (ob < 0) break;
            const R* py = px + ob;
            R s0[A], s1[A];
#pragma unroll
            for (int n = 0; n < A; ++n) s0[n] = py[oz[n].x];
#pragma unroll
            for (int n = 0; n < A; ++n) s1[n] = oz[n].y >= 0 ? py[oz[n].y] : R(0);
#pragma unroll
            for (int n = 0; n < A; ++n) {
                v[n] += s0[n];
                v[n] += s1[n];
            }
            if (ps.deep) {
#pragma unroll
                for (int n = 0; n < A; ++n) {
                    if (SEAM && !near_seam(B * n, B * n + B - 1, A * B)) continue;
                    const int2 d = __ldg(reinterpret_cast<const int2*>(&zoff[B * n]) + 1);
                    if (d.x >= 0) v[n] += py[d.x];
                    if (d.y >= 0) v[n] += py[d.y];
                }
            }
        }
    }
}

// The transform of a pair's rows from the points each thread holds (v[q][n] =
// point B n + j + T q, row 0 + i row 1), and the two half rows out to o0 and
// o0 + Hz (the second if `two`).
template <typename R, int L, int CAP = kPairCap<R>>
__device__ __forceinline__ void z_forward(typename CT<R>::C (&v)[FacZ<L, CAP>::G1][FacZ<L, CAP>::A], bool on, bool two, int j,
                                          typename CT<R>::C* sm, const typename CT<R>::C* __restrict__ tw,
                                          typename CT<R>::C* __restrict__ o0) {
    typedef PairEngine<R, L, CAP> E;
    typedef typename CT<R>::C C;
    constexpr int A = E::A, B = E::B, T = E::T, G1 = E::G1, Hz = L / 2 + 1;
#pragma unroll
    for (int q = 0; q < G1; ++q)
        if (on && j + T * q < B) E::space_out(v[q], j + T * q, sm, tw);
    E::sync();
    if (!on || j >= E::T2) return;
    const int kb1 = pair_k1<A>(j);
    const bool bon = pair_on<A>(j);
    C za[B], zb[B];
    E::spec_in(za, j, sm);
    if (bon) {
        E::spec_in(zb, kb1, sm);
    } else {
#pragma unroll
        for (int k = 0; k < B; ++k) zb[k] = za[k];
    }
    C* o1 = o0 + Hz;
    auto put = [&](int k, C z, C mirror) {  // x0 = (Z + conj Z') / 2, x1 = (Z - conj Z') / 2i
        const C zc = cconj(mirror), d = csub(z, zc);
        o0[k] = cscale(cadd(z, zc), R(0.5));
        if (two) o1[k] = CT<R>::mk(R(0.5) * d.y, R(-0.5) * d.x);
    };
#pragma unroll
    for (int k = 0; k <= B / 2; ++k) {
        // mirror of k1 + A k2: (A - k1) + A (B - 1 - k2), of A k2: A (B - k2)
        const C ma0 = za[(B - k) % B], mb = zb[B - 1 - (k < B ? k : 0)], maj = za[B - 1 - (k < B ? k : 0)];
        const int ka = j + A * k, kb = kb1 + A * k;
        const C ma = j > 0 ? mb : ma0;
        if (ka < Hz) put(ka, za[k % B], ma);
        const C mbb = j > 0 ? maj : mb;
        if (bon && kb < Hz) put(kb, zb[k % B], mbb);
    }
}

// The pass's factors: in FP64 a thread takes one butterfly of lines up to 64.  It
// folds the points of its butterflies one after another, and a 64-point line has
// only four threads at two each: 64^3 25.0 -> 21.3 us (22.4 for the pass staged
// through shared memory).  The inverse keeps two, with which every thread has a
// part of both stages (28.7 us against 41.0).
template <typename R, int L>
constexpr int kFoldCap = sizeof(R) == 8 && L <= 64 ? 8 : kPairCap<R>;
template <typename R, int L>
using FacF = FacZ<L, kFoldCap<R, L>>;

template <typename R, int L, bool SPLIT>
__global__ void __launch_bounds__((SPLIT ? 2 : 1) * FacF<R, L>::T * FacF<R, L>::NPMAX,
                                  SPLIT ? pass_blocks<R, 2 * FacF<R, L>::T * FacF<R, L>::NPMAX>(40 + 7 * FacF<R, L>::G1 * FacF<R, L>::A / 2)
                                        : pass_blocks<R, FacF<R, L>::T * FacF<R, L>::NPMAX>(48 + 5 * FacF<R, L>::G1 * FacF<R, L>::A))
k_fft_z_r2c_reg(Geo g, const typename CT<R>::C* __restrict__ tw, const R* __restrict__ in,
                typename CT<R>::C* __restrict__ out, int rows, PatchSrc<R> ps) {
    pdl_enter();
    typedef PairEngine<R, L, kFoldCap<R, L>> E;
    typedef typename CT<R>::C C;
    constexpr int A = E::A, B = E::B, T = E::T, G1 = E::G1, Hz = L / 2 + 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nt = SPLIT ? blockDim.x / 2 : blockDim.x;  // threads of one set
    const bool odd = SPLIT && (int)threadIdx.x >= nt;
    const int t = odd ? threadIdx.x - nt : threadIdx.x;
    const int p = t / T, j = t - p * T;
    const int pair = blockIdx.x * (nt / T) + p;
    bool on = 2 * pair < rows;
    const int r0 = 2 * pair;
    const bool two = r0 + 1 < rows;
    C* sm = reinterpret_cast<C*>(smem_raw) + p * E::PITCH;
    R* hand = reinterpret_cast<R*>(sm);  // the odd row, point z at hand[z]
    C v[G1][A];
#pragma unroll
    for (int q = 0; q < G1; ++q) {
        const int n2 = j + T * q;
        if (!on || n2 >= B) continue;
        if (ps.patch) {
            R f[A];
            if (!odd || two) {
                fold_row<R, A, B, true>(g, ps, r0 + (odd ? 1 : 0), n2, f);
            } else {
#pragma unroll
                for (int n = 0; n < A; ++n) f[n] = R(0);
            }
#pragma unroll
            for (int n = 0; n < A; ++n) {
                if (odd) hand[B * n + n2] = f[n];
                else v[q][n].x = f[n];
            }
            if constexpr (!SPLIT) {
                if (two) {
                    fold_row<R, A, B, true>(g, ps, r0 + 1, n2, f);
                } else {
#pragma unroll
                    for (int n = 0; n < A; ++n) f[n] = R(0);
                }
#pragma unroll
                for (int n = 0; n < A; ++n) v[q][n].y = f[n];
            }
        } else if (!odd) {
            const R* a0 = in + (int64_t)r0 * L + n2;
#pragma unroll
            for (int n = 0; n < A; ++n) v[q][n] = CT<R>::mk(a0[B * n], two ? a0[L + B * n] : R(0));
        }
    }
    if constexpr (SPLIT) {
        __syncthreads();
        if (odd && E::kWarp) return;
        on &= !odd;  // (the odd rows' threads go on to the block's barriers)
        if (ps.patch) {
#pragma unroll
            for (int q = 0; q < G1; ++q)
                if (on && j + T * q < B)
#pragma unroll
                    for (int n = 0; n < A; ++n) v[q][n].y = hand[B * n + j + T * q];
        }
        E::sync();  // before the line takes the hand-over's space
    }
    z_forward<R, L, kFoldCap<R, L>>(v, on, two, j, sm, tw, out + (int64_t)r0 * Hz);
}

// ------------------------------------------------------------------ z inverse (C2R)
// The half-spectrum values of two real lines (two rows of a field, or two
// fields of a row) joined to one complex line h0 + i h1 on the spectral side.
// mul: multiply by -i kz' first (kz' = 0 on the Nyquist index).
template <typename R, int L>
__device__ __forceinline__ void z_join(const Geo& g, const typename CT<R>::C* __restrict__ h0p, bool mul0,
                                       const typename CT<R>::C* __restrict__ h1p, bool mul1, bool two, int j,
                                       typename CT<R>::C* sm, const typename CT<R>::C* __restrict__ tw) {
    typedef PairEngine<R, L> E;
    typedef typename CT<R>::C C;
    constexpr int A = E::A, B = E::B, Hz = L / 2 + 1, M = B / 2 + 1;
    const int kb1 = pair_k1<A>(j);
    const bool bon = pair_on<A>(j);
    C da[M], ma[M], db[M], mb[M];
    auto get = [&](int k, C& direct, C& mirror) {
        C h0 = h0p[k], h1 = two ? h1p[k] : CT<R>::mk(R(0), R(0));
        const bool real = k == 0 || (L % 2 == 0 && 2 * k == L);
        const R kz = (L % 2 == 0 && 2 * k == L) ? R(0) : kfac<R>(g, 2) * k;
        if (mul0) h0 = CT<R>::mk(kz * h0.y, -kz * h0.x);
        if (mul1) h1 = CT<R>::mk(kz * h1.y, -kz * h1.x);
        if (real) h0.y = h1.y = R(0);
        direct = CT<R>::mk(h0.x - h1.y, h0.y + h1.x);
        mirror = CT<R>::mk(h0.x + h1.y, h1.x - h0.y);
    };
#pragma unroll
    for (int k = 0; k < M; ++k) {
        da[k] = ma[k] = db[k] = mb[k] = CT<R>::mk(R(0), R(0));
        const int ka = j + A * k, kb = kb1 + A * k;
        if (ka < Hz) get(ka, da[k], ma[k]);
        if (bon && kb < Hz) get(kb, db[k], mb[k]);
    }
    C za[B], zb[B];
#pragma unroll
    for (int k = 0; k < B; ++k) {
        // upper half from the mirrors: of k2 it is B - 1 - k2 of the other
        // frequency, for frequency 0 its own B - k2, for A / 2 its own B - 1 - k2
        if (2 * k + 1 < B) {
            za[k] = da[k];
            zb[k] = db[k];
        } else if (2 * k + 1 == B) {
            za[k] = da[k];
            zb[k] = j > 0 ? ma[k] : db[k];
        } else {
            za[k] = j > 0 ? mb[B - 1 - k] : ma[B - k];
            zb[k] = j > 0 ? ma[B - 1 - k] : mb[B - 1 - k];
        }
    }
    E::spec_out(za, j, sm, tw);
    if (bon) E::spec_out(zb, kb1, sm, tw);
}

// store(o) for the offset o of row r of the padded layout and of each of its
// periodic images (at most one per axis: Xp < 2 Nx)
template <typename F>
__device__ __forceinline__ void row_images(const Geo& g, const FieldLayout& fl, int r, F store) {
    const int Nx = g.N[0], Ny = g.N[1], kmin = g.kmin;
    const int x = r / Ny, y = r - x * Ny;
    const int px0 = x - kmin, py0 = y - kmin;
    const int pxg = px0 + Nx < fl.Xp ? px0 + Nx : (px0 - Nx >= 0 ? px0 - Nx : -1);
    const int pyg = py0 + Ny < fl.Yp ? py0 + Ny : (py0 - Ny >= 0 ? py0 - Ny : -1);
#pragma unroll 1
    for (int im = 0; im < 4; ++im) {
        const int px = (im & 1) ? pxg : px0, py = (im & 2) ? pyg : py0;
        if (px >= 0 && py >= 0) store(((int64_t)px * fl.Yp + py) * fl.Zp);
    }
}

// Point B n + n2 of a line of L to out[o + its padded z] and to its z ghost (only
// the first and last few points have one); n is a constant where it is called.
template <int L, int B, typename V>
__device__ __forceinline__ void put_point(V* out, int64_t o, int n, int n2, int kmin, int Zp, V val) {
    const int pz = B * n + n2 - kmin;
    out[o + pz] = val;
    if (B * n < kMaxOrder && pz + L < Zp) out[o + pz + L] = val;
    if (B * (n + 1) > L - kMaxOrder && pz >= L) out[o + pz - L] = val;
}

// One field (blockIdx.y) into an unpadded mesh, two rows a line.
template <typename R, int L>
__global__ void __launch_bounds__(FacI<R, L>::T * FacI<R, L>::NPMAX)
k_fft_z_c2r_plain(Geo g, const typename CT<R>::C* __restrict__ tw, ZOut zo, int rows) {
    pdl_enter();
    typedef PairEngine<R, L> E;
    typedef typename CT<R>::C C;
    constexpr int A = E::A, B = E::B, T = E::T, Hz = L / 2 + 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int p = threadIdx.x / T, j = threadIdx.x - p * T;
    const int pair = blockIdx.x * (blockDim.x / T) + p, f = blockIdx.y;
    const bool on = 2 * pair < rows, two = 2 * pair + 1 < rows;
    C* sm = reinterpret_cast<C*>(smem_raw) + p * E::PITCH;
    if (on && j < E::T2) {
        const C* h = reinterpret_cast<const C*>(pick4(zo.src, f)) + (int64_t)(2 * pair) * Hz;
        const bool mul = pick4(zo.mulkz, f) != 0;
        z_join<R, L>(g, h, mul, h + Hz, mul, two, j, sm, tw);
    }
    E::sync();
    if (!on) return;
    R* out = reinterpret_cast<R*>(pick4(zo.out, f)) + (int64_t)(2 * pair) * L;
#pragma unroll
    for (int q = 0; q < E::G1; ++q) {
        const int n2 = j + T * q;
        if (n2 < B) {
            C v[A];
            E::space_in(v, n2, sm);
#pragma unroll
            for (int n = 0; n < A; ++n) {
                out[B * n + n2] = v[n].x;
                if (two) out[L + B * n + n2] = v[n].y;
            }
        }
    }
}

// All fields of two rows into the padded mesh, one set of T threads a line:
// set 0 of a pair transforms E_z of both rows, sets 1 and 2 E_x and E_y of one
// row each; set 0 hands E_z over through shared memory and the others store a
// point's three fields with one 16-byte store (32 bytes in FP64) to the row,
// to its periodic images and to the z ghosts.  With the potential as a fourth
// output a set 3 transforms both rows of it.
template <typename R, int L>
constexpr size_t c2r_pair_bytes(int nf) {
    return sizeof(typename CT<R>::C) * FacI<R, L>::PITCH * nf + 2 * L * sizeof(R) + (L % 2) * 2 * sizeof(R);
}
template <typename R, int L>
struct FacC2R {  // pairs a block holds at most at three lines a pair, about 192 threads
    typedef FacI<R, L> F;
    static constexpr int NPMAX = F::T <= 32 ? 64 / F::T : 2, NT = 3 * F::T * NPMAX;
    static constexpr int PTS = F::G1 * F::A > 2 * F::B ? F::G1 * F::A : 2 * F::B;
};

template <typename R, int L>
__global__ void __launch_bounds__(FacC2R<R, L>::NT, pass_blocks<R, FacC2R<R, L>::NT>(32 + 3 * FacC2R<R, L>::PTS))
k_fft_z_c2r_reg(Geo g, const typename CT<R>::C* __restrict__ tw, ZOut zo, int rows) {
    pdl_enter();
    typedef PairEngine<R, L> E;
    typedef typename CT<R>::C C;
    typedef typename CT<R>::C4 V4;
    constexpr int A = E::A, B = E::B, T = E::T, G1 = E::G1, Hz = L / 2 + 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nf = zo.nf, np = blockDim.x / (nf * T);
    const int line = threadIdx.x / T, j = threadIdx.x - line * T;
    const int p = line / nf, set = line - p * nf;
    const int pair = blockIdx.x * np + p;
    const bool on = 2 * pair < rows, two = 2 * pair + 1 < rows;
    C* sm = reinterpret_cast<C*>(smem_raw) + line * E::PITCH;
    R* ez = reinterpret_cast<R*>(reinterpret_cast<C*>(smem_raw) + np * nf * E::PITCH) + p * (2 * L);
    const bool ron = on && (set != 2 || two);
    if (ron && j < E::T2) {
        const int64_t r0 = (int64_t)(2 * pair) * Hz;
        const bool row = set == 1 || set == 2;
        const C* h0 = reinterpret_cast<const C*>(row ? zo.src[0] : zo.src[2]) + r0 + (set == 2 ? Hz : 0);
        const C* h1 = row ? reinterpret_cast<const C*>(zo.src[1]) + r0 + (set == 2 ? Hz : 0) : h0 + Hz;
        z_join<R, L>(g, h0, set == 0, h1, set == 0, row || two, j, sm, tw);
    }
    E::sync();
    C v[G1][A];
#pragma unroll
    for (int q = 0; q < G1; ++q) {
        const int n2 = j + T * q;
        if (ron && n2 < B) {
            E::space_in(v[q], n2, sm);
            if (set == 0) {
#pragma unroll
                for (int n = 0; n < A; ++n) {
                    ez[B * n + n2] = v[q][n].x;
                    ez[L + B * n + n2] = v[q][n].y;
                }
            }
        }
    }
    __syncthreads();
    if (!ron || set == 0) return;
    const FieldLayout& fl = zo.fl;
    if (set == 3) {
        R* phi = reinterpret_cast<R*>(zo.out[3]);
#pragma unroll 1
        for (int half = 0; half < (two ? 2 : 1); ++half)
            row_images(g, fl, 2 * pair + half, [&](int64_t o) {
#pragma unroll
                for (int q = 0; q < G1; ++q)
#pragma unroll
                    for (int n = 0; n < A; ++n)
                        if (j + T * q < B)
                            put_point<L, B>(phi, o, n, j + T * q, g.kmin, fl.Zp, half ? v[q][n].y : v[q][n].x);
            });
        return;
    }
    V4* out = reinterpret_cast<V4*>(zo.out[0]);
    const R* ezr = ez + (set - 1) * L;
    row_images(g, fl, 2 * pair + set - 1, [&](int64_t o) {
#pragma unroll
        for (int q = 0; q < G1; ++q)
#pragma unroll
            for (int n = 0; n < A; ++n)
                if (j + T * q < B)
                    put_point<L, B>(out, o, n, j + T * q, g.kmin, fl.Zp,
                                    CT<R>::mk4(v[q][n].x, v[q][n].y, ezr[B * n + j + T * q], R(0)));
    });
}

}  // namespace pppm
