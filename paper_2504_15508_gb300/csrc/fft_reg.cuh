// Register-resident line FFTs of the single-box passes.
//
// A line of L = A B points is transformed as n = B n1 + n2, k = k1 + A k2: a
// DFT of A points over n1 for each n2, the twiddle e^{-2 pi i n2 k1 / L}, and a
// DFT of B points over n2 for each k1.  Each DFT is one thread's registers, so
// a transform crosses shared memory once (between its two halves) where a
// Stockham pass that stages its input and output crosses it three times, and
// points go straight between global memory and registers.  The inverse runs
// the same steps backwards (B over k2, twiddle, A over k1), so that a thread
// can go from the forward transform's outputs to the inverse's inputs without
// moving them: that is how the x pass applies the influence function and how
// the z passes pair Hermitian modes.
//
// Measured against Stockham passes in shared memory with the same fusions
// (CUDA events around a launch, about 3 us of each figure is theirs):
//
//   pass                  128^3 FP32     160^3 FP32     64^3 FP64
//   z forward with fold   24.6 -> 16.7   45.0 -> 25.6   22.5 -> 21.4 us
//   y forward             10.2 ->  9.8   15.2 -> 12.7   14.3 -> 11.1
//   x and influence       25.8 -> 12.9   45.0 -> 22.3   73.6 -> 34.9
//   y inverse, 3 outputs  16.8 -> 13.7   29.2 -> 20.1   30.6 -> 22.6
//   z inverse, 3 outputs  24.5 -> 18.0   45.0 -> 35.3   34.8 -> 28.8
//
// and 45 x 60 x 75, lengths that had only a run-time engine: 65.3 -> 42.0 us for
// the five with the fold.  The strided passes are bound by the latency of
// their two global transfers around one exchange, the z passes by their
// patch reads and field writes; FP64 by its arithmetic, at 1/64 of the FP32
// rate.
//
// Every index is a compile-time constant apart from the thread's own.  The
// lengths with an engine are listed in PPPM_REG_LENGTHS; the run-time radix
// passes serve the others.
#pragma once

#include <utility>

#include "fft_common.cuh"

namespace pppm {

// ------------------------------------------------------------------ roots of unity
// cos and sin of 2 pi n / d, reduced to an angle of at most pi / 4 and summed
// as Taylor series in FP64 at compile time.
constexpr double turn_sin(int n, int d);
constexpr double turn_cos(int n, int d) {
    n %= d;
    if (2 * n > d) n = d - n;
    if (4 * n > d) return -turn_cos(d - 2 * n, 2 * d);
    if (8 * n > d) return turn_sin(d - 4 * n, 4 * d);
    const double x = 6.283185307179586476925 * n / d;
    double t = 1.0, s = 1.0;
    for (int k = 1; k < 12; ++k) {
        t *= -x * x / ((2 * k - 1) * (2 * k));
        s += t;
    }
    return s;
}
constexpr double turn_sin(int n, int d) {
    n %= d;
    if (2 * n > d) return -turn_sin(d - n, d);
    if (4 * n > d) return turn_sin(d - 2 * n, 2 * d);
    if (8 * n > d) return turn_cos(d - 4 * n, 4 * d);
    const double x = 6.283185307179586476925 * n / d;
    double t = x, s = x;
    for (int k = 1; k < 12; ++k) {
        t *= -x * x / ((2 * k) * (2 * k + 1));
        s += t;
    }
    return s;
}

template <int N, int M>
struct Root {
    static constexpr double c = turn_cos(M, N), s = turn_sin(M, N);
};

template <int N, typename F, int... I>
__device__ __forceinline__ void static_for_impl(F&& f, std::integer_sequence<int, I...>) {
    (f(std::integral_constant<int, I>{}), ...);
}
template <int N, typename F>
__device__ __forceinline__ void static_for(F&& f) {
    static_for_impl<N>(f, std::make_integer_sequence<int, N>{});
}

// ------------------------------------------------------------------ DFTs in registers
// first factor of a composite size (the second is N / it); 0 for the base sizes
constexpr int dft_split(int N) {
    return N == 6 ? 3 : N == 8 ? 4 : N == 9 ? 3 : N == 10 ? 5 : N == 12 ? 4 : N == 15 ? 5 : N == 16 ? 4
         : N == 18 ? 6 : N == 20 ? 5 : N == 24 ? 6 : N == 25 ? 5 : N == 27 ? 9 : 0;
}
constexpr bool dft_size(int N) { return (N >= 2 && N <= 5) || dft_split(N) > 0; }

// X[k] = sum_n v[n] e^{SIGN 2 pi i n k / N}, in place, natural order
template <typename C, typename R, int N, int SIGN>
__device__ __forceinline__ void dft(C (&v)[N]) {
    if constexpr (dft_split(N) == 0) {
        butterfly<C, R>(v, N, R(SIGN));
    } else {
        constexpr int A = dft_split(N), B = N / A;
        C t[B][A];
        static_for<B>([&](auto n2) {
#pragma unroll
            for (int n1 = 0; n1 < A; ++n1) t[n2][n1] = v[B * n1 + n2];
            dft<C, R, A, SIGN>(t[n2]);
            static_for<A>([&](auto k1) {
                constexpr int m = (decltype(n2)::value * decltype(k1)::value) % N;
                if constexpr (m > 0) {
                    if constexpr (4 * m == N) {  // a quarter turn: no arithmetic
                        t[n2][k1] = cmul_is(t[n2][k1], R(SIGN));
                    } else {
                        t[n2][k1] = cmul(t[n2][k1], CT<R>::mk(R(Root<N, m>::c), R(SIGN * Root<N, m>::s)));
                    }
                }
            });
        });
        static_for<A>([&](auto k1) {
            C u[B];
#pragma unroll
            for (int n2 = 0; n2 < B; ++n2) u[n2] = t[n2][k1];
            dft<C, R, B, SIGN>(u);
#pragma unroll
            for (int k2 = 0; k2 < B; ++k2) v[k1 + A * k2] = u[k2];
        });
    }
}

// ------------------------------------------------------------------ factors of a length
// Strided lines (x and y): 16 lines side by side, T threads a line.  A is the
// smallest usable factor with A >= B; stage 1 has B butterflies of A points
// and stage 2 has A of B points, so T = B threads when B divides A (each runs
// A / B of stage 2: both stages keep every thread busy with at most A points),
// else T = A (one butterfly of either stage a thread).
constexpr int strided_a(int L) {
    for (int a = 2; a <= 27; ++a)
        if (L % a == 0 && a * a >= L && dft_size(a) && dft_size(L / a)) return a;
    return 0;
}
template <int L>
struct FacS {
    static constexpr int A = strided_a(L), B = L / A;
    static constexpr int T = A % B == 0 ? B : A, G2 = A / T, NT = 16 * T;
};

// Contiguous lines (z): two real rows a complex line; a thread of stage 2 holds
// the frequencies k1 and A - k1 (the first one 0 and A / 2), with which every
// mode and its Hermitian mirror lie in one thread.  A is chosen for the
// fewest points a thread, max(A, 2 B), then for an even A.  A thread takes several
// butterflies of stage 1 where that gives both stages the same threads and is no
// more than CAP points.
constexpr int paired_a(int L, int cap) {
    int best = 0, cost = 1 << 30;
    for (int a = 2; a <= 27; ++a) {
        if (L % a != 0 || !dft_size(a) || !dft_size(L / a)) continue;
        const int b = L / a, t2 = a / 2 + a % 2, e = a > 2 * b ? a : 2 * b;
        const int t = b % t2 == 0 && (b / t2) * a <= cap ? t2 : (t2 > b ? t2 : b);
        const int c = 64 * e + 32 * (a % 2) + t;
        if (c < cost) {
            cost = c;
            best = a;
        }
    }
    return best;
}
template <int L, int CAP = 16>
struct FacZ {
    static constexpr int A = paired_a(L, CAP), B = L / A;
    static constexpr int T2 = A / 2 + A % 2;  // threads of stage 2
    static constexpr int T = B % T2 == 0 && (B / T2) * A <= CAP ? T2 : (T2 > B ? T2 : B);
    static constexpr int G1 = T < B ? B / T : 1;  // butterflies of stage 1 a thread
    static constexpr bool kWarp = 32 % T == 0;    // a line's threads share a warp
    // lines a block holds at most: about 128 threads, whole warps where T allows
    static constexpr int NPMAX = T <= 128 ? 128 / T : 1;
    // shared-memory pitch of a line: rows k1 of B + 1 values, and the lines of
    // a warp T values apart in the banks
    static constexpr int P0 = A * (B + 1);
    static constexpr int PITCH = P0 + ((T - P0) % 16 + 16) % 16;
};

// Points a thread of the z passes takes at most as several butterflies.  FP64: with
// one butterfly a thread half the threads of a 100-point line have no part in stage
// 2, and the line's ten do not share a warp: 100^3 z forward 77 -> 61 us, inverse
// 172 -> 121.
template <typename R>
constexpr int kPairCap = sizeof(R) == 8 ? 20 : 16;
template <typename R, int L>
using FacI = FacZ<L, kPairCap<R>>;

// the lengths served by the register engines
#define PPPM_REG_LENGTHS(X)                                                                                   \
    X(8) X(9) X(10) X(12) X(15) X(16) X(18) X(20) X(24) X(25) X(27) X(30) X(32) X(36) X(40) X(45) X(48) X(50) \
    X(54) X(60) X(64) X(72) X(75) X(80) X(81) X(90) X(96) X(100) X(108) X(120) X(125) X(128) X(135) X(144)    \
    X(150) X(160) X(162) X(180) X(192) X(200) X(216) X(225) X(240) X(250) X(256)

// FP64 plans: shorter lines (a thread's points take twice the registers)
#define PPPM_REG_LENGTHS_F64(X)                                                                               \
    X(8) X(9) X(10) X(12) X(15) X(16) X(18) X(20) X(24) X(25) X(27) X(30) X(32) X(36) X(40) X(45) X(48) X(50) \
    X(54) X(60) X(64) X(72) X(75) X(80) X(81) X(90) X(96) X(100) X(108) X(120) X(128)

// resident blocks per SM of a kernel (0: it does not fit)
template <typename K>
int resident_blocks(K kern, int threads, size_t smem) {
    int per = 0;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, threads, smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return per;
}

// Blocks of NT threads an SM should hold when a thread may take `regs`
// registers (a pass's fixed needs plus its points): the launch bound of the
// FP32 kernels.  FP64 kernels are not limited: their arithmetic, at a small
// fraction of the FP32 rate, is far slower than the issue of anything else.
template <typename R, int NT>
constexpr int pass_blocks(int regs) {
    return sizeof(R) != 4 || 65536 / (NT * regs) < 1 ? 1 : 65536 / (NT * regs);
}

// twiddle e^{SIGN 2 pi i m / L} from the table of e^{-2 pi i m / L}
template <typename R, int SIGN>
__device__ __forceinline__ typename CT<R>::C twiddle(const typename CT<R>::C* __restrict__ tw, int m) {
    typename CT<R>::C w = __ldg(&tw[m]);
    if (SIGN > 0) w.y = -w.y;
    return w;
}

}  // namespace pppm
