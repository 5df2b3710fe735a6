// The FFT stages of the batched form's staged launch on the register engines
// (fft_reg.cuh, fft_xy.cuh, fft_z.cuh): each stage one kernel over that stage's
// items of every box, a block's item chosen from the list, its line length by
// a switch (all lengths up to 64, the batch's meshes; a batch with longer lines
// runs the general stages).
//
// Against the general stages, whose lines are staged through shared memory
// before and after a Stockham FFT there, with run-time index arithmetic and a
// fold of up to 64 predicated loads a point (96 boxes of 64-8,192 molecules,
// 1.9 M half-spectrum points, ncu): z forward 122.6 -> 37.3 us, y forward
// 33.6 -> 18.0, x 106.1 -> 42.8, y inverse 76.1 -> 30.6, z inverse 119.2 -> 47.2;
// the batch 710 -> 449 us.
#include "batched.cuh"
#include "fft_xy.cuh"
#include "fft_z.cuh"

namespace pppm {
namespace batch {

#define PPPM_BATCH_LENGTHS(X)                                                                                 \
    X(6) X(8) X(9) X(10) X(12) X(15) X(16) X(18) X(20) X(24) X(25) X(27) X(30) X(32) X(36) X(40) X(45) X(48)  \
    X(50) X(54) X(60) X(64)

// lines of an item, and its shared memory
template <int L>
struct Strided {
    static constexpr int NG = kThreads / FacS<L>::NT, LINES = 16 * NG;  // groups of 16 lines
};
template <int L>
struct Contig {
    static constexpr int LINES = kThreads / FacZ<L>::T;
};

template <int L>
constexpr size_t smem_of(int stage) {
    const size_t strided = sizeof(float2) * L * 16 * Strided<L>::NG, contig = sizeof(float2) * FacZ<L>::PITCH * Contig<L>::LINES;
    const size_t red = 7 * sizeof(float) * kThreads;
    return stage == S_YFWD ? strided
         : stage == S_YINV ? 2 * strided
         : stage == S_XINF ? (2 * strided > red ? 2 * strided : red)
                           : contig;
}

template <int L>
int items_of(int stage, int64_t lines) {
    const int per = stage == S_ZR2C || stage == S_ZC2R ? Contig<L>::LINES : Strided<L>::LINES;
    return (int)((lines + per - 1) / per);
}

// the axis a stage transforms, and the lines of a box
static int stage_axis(int stage) { return stage == S_ZR2C || stage == S_ZC2R ? 2 : stage == S_XINF ? 0 : 1; }
static int64_t stage_lines(int stage, const int N[3], int Hz) {
    const int64_t pairs = ((int64_t)N[0] * N[1] + 1) / 2;
    switch (stage) {
        case S_ZR2C: return pairs;
        case S_ZC2R: return 3 * pairs;  // a line a field
        case S_XINF: return (int64_t)N[1] * Hz;
        default: return (int64_t)N[0] * Hz;
    }
}

// line of a strided item: this thread's group, column and place in the line
template <int L>
struct Place {
    int grp, l, j;
    int64_t f;
    __device__ __forceinline__ Place(int idx) {
        grp = threadIdx.x / FacS<L>::NT;
        const int t = threadIdx.x - grp * FacS<L>::NT;
        l = t & 15;
        j = t >> 4;
        f = (int64_t)idx * Strided<L>::LINES + grp * 16 + l;
    }
    __device__ __forceinline__ bool on(int64_t lines) const { return grp < Strided<L>::NG && f < lines; }
};

template <int L>
__device__ __forceinline__ void run_z_r2c(const BoxDesc& D, int idx, const Bufs& B, unsigned char* smem) {
    typedef FacZ<L> F;
    const Geo& g = D.g;
    const int rows = g.N[0] * g.N[1];
    const int p = threadIdx.x / F::T, j = threadIdx.x - p * F::T;
    const int pair = idx * Contig<L>::LINES + p;
    const bool on = p < Contig<L>::LINES && 2 * pair < rows, two = 2 * pair + 1 < rows;
    PatchSrc<float> ps;
    ps.patch = B.patch + D.patch0;
    ps.cov = B.cov_x + D.cov_x0;
    ps.off = B.cov_yz + D.cov_yz0;
    ps.nmax = D.nmax;
    ps.deep = D.cov_deep;
    ps.xstride = D.xstride;
    float2 v[F::G1][F::A];
#pragma unroll
    for (int q = 0; q < F::G1; ++q) {
        const int n2 = j + F::T * q;
        if (!on || n2 >= F::B) continue;
        float f[F::A];
        fold_row<float, F::A, F::B, false>(g, ps, 2 * pair, n2, f);
#pragma unroll
        for (int n = 0; n < F::A; ++n) v[q][n] = make_float2(f[n], 0.f);
        if (two) {
            fold_row<float, F::A, F::B, false>(g, ps, 2 * pair + 1, n2, f);
#pragma unroll
            for (int n = 0; n < F::A; ++n) v[q][n].y = f[n];
        }
    }
    z_forward<float, L>(v, on, two, j, reinterpret_cast<float2*>(smem) + p * F::PITCH, B.tw + D.tw0[2],
                        B.cx0 + D.c0 + (int64_t)(2 * pair) * (L / 2 + 1));
}

template <int L>
__device__ __forceinline__ void run_y(const BoxDesc& D, int idx, const Bufs& B, unsigned char* smem) {
    const int Hz = D.g.Hz;
    const Place<L> a(idx);
    float2* sm = reinterpret_cast<float2*>(smem) + a.grp * (L * 16) + a.l;
    line_body<float, L, -1>(a.on((int64_t)D.g.N[0] * Hz), a.j, sm, B.tw + D.tw0[1],
                            B.cx0 + D.c0 + (a.f / Hz) * ((int64_t)L * Hz) + a.f % Hz, Hz);
}

// the last item of a box sums that box's partials
template <int L>
__device__ __forceinline__ void run_x(const BoxDesc& D, int box, int idx, const Bufs& B, unsigned char* smem) {
    const int Hz = D.g.Hz;
    const int64_t es = (int64_t)D.g.N[1] * Hz;
    const Place<L> a(idx);
    float2* s0 = reinterpret_cast<float2*>(smem) + a.grp * (2 * L * 16) + a.l;
    const int y = (int)(a.f / Hz), kz = (int)(a.f - (int64_t)y * Hz);
    float term[7];
    x_body<float, L>(a.on(es), a.j, s0, s0 + L * 16, B.tw + D.tw0[0], B.G + D.G0 + a.f, B.cx0 + D.c0 + a.f,
                     B.cx1 + D.c0 + a.f, es, x_line<float>(D.g, y, kz, D.beta, D.e_scale, D.c_field), term);
    __syncthreads();
    block_terms<float, kThreads>(term, reinterpret_cast<float*>(smem), B.partial + (int64_t)(D.part0 + idx) * 14);
    __threadfence();
    __syncthreads();
    __shared__ bool last;
    if (threadIdx.x == 0)
        last = atomicAdd(&B.box_counter[box], 1u) == (unsigned)D.rnitems[S_XINF - S_ZR2C] - 1;
    __syncthreads();
    if (last) {
        __threadfence();
        finish_energy(B.partial + (int64_t)D.part0 * 14, D.rnitems[S_XINF - S_ZR2C], B.prefactor, B.energy + box,
                      B.virial + 6 * box);
    }
}

template <int L>
__device__ __forceinline__ void run_y_inv(const BoxDesc& D, int idx, const Bufs& B, unsigned char* smem) {
    const int Hz = D.g.Hz;
    const Place<L> a(idx);
    float2* s0 = reinterpret_cast<float2*>(smem) + a.grp * (2 * L * 16) + a.l;
    const int64_t off = D.c0 + (a.f / Hz) * ((int64_t)L * Hz) + a.f % Hz;
    y_inv3_body<float, L>(a.on((int64_t)D.g.N[0] * Hz), a.j, s0, s0 + L * 16, B.tw + D.tw0[1], D.g.kfac_f[1],
                          B.cx0 + off, B.cx1 + off, B.cx2 + off, Hz);
}

// one field of two rows a line, into the planar padded fields
template <int L>
__device__ __forceinline__ void run_z_c2r(const BoxDesc& D, int idx, const Bufs& B, unsigned char* smem) {
    typedef PairEngine<float, L> E;
    const Geo& g = D.g;
    const int rows = g.N[0] * g.N[1], pairs = (rows + 1) / 2;
    const int line = threadIdx.x / E::T, j = threadIdx.x - line * E::T;
    const int gl = idx * Contig<L>::LINES + line;
    const int pair = gl / 3, f = gl - 3 * pair;
    const bool on = line < Contig<L>::LINES && pair < pairs, two = 2 * pair + 1 < rows;
    float2* sm = reinterpret_cast<float2*>(smem) + line * E::PITCH;
    if (on && j < E::T2) {
        const float2* src = f == 0 ? B.cx1 : f == 1 ? B.cx2 : B.cx0;
        const float2* h = src + D.c0 + (int64_t)(2 * pair) * (L / 2 + 1);
        z_join<float, L>(g, h, f == 2, h + (L / 2 + 1), f == 2, two, j, sm, B.tw + D.tw0[2]);
    }
    E::sync();
    if (!on) return;
    float2 v[E::G1][E::A];
#pragma unroll
    for (int q = 0; q < E::G1; ++q)
        if (j + E::T * q < E::B) E::space_in(v[q], j + E::T * q, sm);
    float* out = B.fields + D.f0 + f * D.fl.fstride;
#pragma unroll 1
    for (int half = 0; half < (two ? 2 : 1); ++half)
        row_images(g, D.fl, 2 * pair + half, [&](int64_t o) {
#pragma unroll
            for (int q = 0; q < E::G1; ++q)
#pragma unroll
                for (int n = 0; n < E::A; ++n)
                    if (j + E::T * q < E::B)
                        put_point<L, E::B>(out, o, n, j + E::T * q, g.kmin, D.fl.Zp, half ? v[q][n].y : v[q][n].x);
        });
}

template <int STAGE, int L>
__device__ __forceinline__ void run_fft(const BoxDesc& D, int box, int idx, const Bufs& B, unsigned char* smem) {
    if constexpr (STAGE == S_ZR2C) run_z_r2c<L>(D, idx, B, smem);
    if constexpr (STAGE == S_YFWD) run_y<L>(D, idx, B, smem);
    if constexpr (STAGE == S_XINF) run_x<L>(D, box, idx, B, smem);
    if constexpr (STAGE == S_YINV) run_y_inv<L>(D, idx, B, smem);
    if constexpr (STAGE == S_ZC2R) run_z_c2r<L>(D, idx, B, smem);
}

template <int STAGE>
__global__ void __launch_bounds__(kThreads, 3)  // 85 registers
k_fft_stage(const BoxDesc* __restrict__ boxes, const int2* __restrict__ items, Bufs B) {
    pdl_enter();
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(16) BoxDesc D;
    const int2 I = items[blockIdx.x];
    {
        const int* src = reinterpret_cast<const int*>(boxes + I.x);
        int* dst = reinterpret_cast<int*>(&D);
        for (int w = threadIdx.x; w < (int)(sizeof(BoxDesc) / sizeof(int)); w += kThreads) dst[w] = src[w];
    }
    __syncthreads();
    switch (D.g.N[STAGE == S_ZR2C || STAGE == S_ZC2R ? 2 : STAGE == S_XINF ? 0 : 1]) {
#define PPPM_LEN(L) \
    case L: run_fft<STAGE, L>(D, I.x, I.y, B, smem); break;
        PPPM_BATCH_LENGTHS(PPPM_LEN)
#undef PPPM_LEN
    }
}

bool reg_fft_length(int L) {
    switch (L) {
#define PPPM_LEN(LL) case LL:
        PPPM_BATCH_LENGTHS(PPPM_LEN)
#undef PPPM_LEN
        return true;
    }
    return false;
}

int reg_fft_items(int stage, const int N[3], int Hz) {
    const int64_t lines = stage_lines(stage, N, Hz);
    switch (N[stage_axis(stage)]) {
#define PPPM_LEN(L) \
    case L: return items_of<L>(stage, lines);
        PPPM_BATCH_LENGTHS(PPPM_LEN)
#undef PPPM_LEN
    }
    return 0;
}

size_t reg_fft_smem(int stage, const int N[3]) {
    switch (N[stage_axis(stage)]) {
#define PPPM_LEN(L) \
    case L: return smem_of<L>(stage);
        PPPM_BATCH_LENGTHS(PPPM_LEN)
#undef PPPM_LEN
    }
    return 0;
}

template <int STAGE>
static cudaError_t launch_stage(cudaStream_t s, const BoxDesc* boxes, const int2* items, int count, const Bufs& B,
                                size_t smem) {
    auto kern = k_fft_stage<STAGE>;
    const cudaError_t e = allow_smem(kern, smem);
    if (e != cudaSuccess) return e;
    return launch_k(kern, dim3(count), dim3(kThreads), smem, s, boxes, items, B);
}

cudaError_t launch_reg_fft(cudaStream_t s, int stage, const BoxDesc* boxes, const int2* items, int count,
                           const Bufs& B, size_t smem) {
    if (count == 0) return cudaSuccess;
    switch (stage) {
        case S_ZR2C: return launch_stage<S_ZR2C>(s, boxes, items, count, B, smem);
        case S_YFWD: return launch_stage<S_YFWD>(s, boxes, items, count, B, smem);
        case S_XINF: return launch_stage<S_XINF>(s, boxes, items, count, B, smem);
        case S_YINV: return launch_stage<S_YINV>(s, boxes, items, count, B, smem);
        case S_ZC2R: return launch_stage<S_ZC2R>(s, boxes, items, count, B, smem);
    }
    return cudaErrorInvalidValue;
}

}  // namespace batch
}  // namespace pppm
