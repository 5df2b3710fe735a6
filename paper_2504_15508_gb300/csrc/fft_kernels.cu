// Mixed-radix (2, 3, 4, 5) 3D FFT passes of the PPPM path, and the fused
// influence-function pass.
//
// Layout: real meshes are Nx x Ny x Nz (z fastest); spectra are half spectra
// Nx x Ny x Hz complex, Hz = Nz/2 + 1, in the same order.
//
// Every pass moves a batch of 1D lines into shared memory, transforms them
// with a self-sorting (Stockham) mixed-radix FFT between two shared buffers,
// and writes them back:
//   z forward   real rows, two per complex FFT (a + i b), unpacked to two half rows;
//   y, x        strided lines, B consecutive (outer, kz) lines per block;
//   x + G       forward x FFT, multiply by the influence function with the
//               energy/virial reduction, and the inverse x FFTs of G rho and
//               -i kx G rho in one block (Poisson-ik, Section 3.1 of the paper);
//   y inverse   of G rho and -i ky G rho (after x) and of -i kx G rho;
//   z inverse   Hermitian half rows of two rows (or two fields) packed as a + i b.
// Twiddles come from a table of e^{-2 pi i t / L} built on the device in FP64
// with sincospi and rounded to the mesh precision.
//
// The kernels here serve any 2^a 3^b 5^c length (radix plan read at run time);
// those from 8 to 256 but 243 (FP64: to 128 but 125) run the same passes on the
// register engines instead (fft_reg.cuh, fft_xy.cuh, fft_z.cuh), a line's points
// in registers with every index and radix a compile-time constant.
#include <atomic>

#include "fft_xy.cuh"
#include "internal.cuh"

namespace pppm {

int device_sms() {
    static std::atomic<int> sms[kResidentCacheDevices];  // 0: not asked yet
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return 1;
    if (dev < kResidentCacheDevices && (n = sms[dev].load(std::memory_order_relaxed)) > 0) return n;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) return 1;
    if (dev < kResidentCacheDevices) sms[dev].store(n, std::memory_order_relaxed);
    return n;
}

template <typename R>
struct GenEngine {
    typedef typename CT<R>::C C;
    Radix rp;
    const C* tw;
    __device__ __forceinline__ int len() const { return rp.L; }
    template <int SIGN, bool LF>
    __device__ __forceinline__ C* run(C* a, C* b, int nl, int ls, int ps) const {
        return stockham<R>(a, b, nl, ls, ps, rp, tw, R(SIGN), LF);
    }
};

template <typename K>
cudaError_t set_smem(K kernel, size_t smem) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

// 2D loop helpers for the bundle kernels: rows of the line (t) by 16-lane groups,
// lines (l) by lane within the group.
#define BUNDLE_LOOP(t, l, L_, nl_)                                              \
    _Pragma("unroll") for (int t = threadIdx.x >> 4; t < (L_); t += kFftThreads >> 4) \
        for (int l = threadIdx.x & 15; l < (nl_); l += 16)
// line-major loops for the z passes: lines by warp, points by lane
#define LINE_LOOP(line, t, nlines_, len_)                                       \
    for (int line = threadIdx.x >> 5; line < (nlines_); line += kFftThreads >> 5) \
        _Pragma("unroll") for (int t = threadIdx.x & 31; t < (len_); t += 32)

// ------------------------------------------------------------------ z forward (R2C)
// Sums of the tile patches covering the points z0, z0 + 32, .. of row (x, y) (the
// fold of the atomics-free spread) in a fixed order; 0 from point Nz on.  The
// row's x and y entries are the same for the whole warp, and a round of loads
// covers NP points of one (x, y) pair of covers.  Whole z forward passes with
// this fold, with up to 64 predicated loads a point (the entries of every slot
// read again for each), and with a fold kernel and a mesh between where a
// length is ragged (243, 150) and eight predicated loads a point where not:
//   FP32  288^3 244, 508, 382 us   320^3 277, 636, 481   64 x 64 x 288 27, 39, 35
//         243^3 171, 408, 240      32 x 32 x 243 22, 54, 27
//   FP64  144^3 162, 302, 173      192^3 356, 624, 412   64 x 64 x 150 48, 75, 46 us
template <typename R, int NP>
__device__ __forceinline__ void fold_points(const Geo& g, const PatchSrc<R>& ps, int row, int z0, int Nz, R (&v)[NP]) {
    const int4* zoff = ps.off + ps.nmax + z0;
    int2 oz[NP];
#pragma unroll
    for (int n = 0; n < NP; ++n) {
        oz[n] = z0 + 32 * n < Nz ? __ldg(reinterpret_cast<const int2*>(&zoff[32 * n])) : make_int2(-1, -1);
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
            R s0[NP], s1[NP];
#pragma unroll
            for (int n = 0; n < NP; ++n) s0[n] = oz[n].x >= 0 ? py[oz[n].x] : R(0);
#pragma unroll
            for (int n = 0; n < NP; ++n) s1[n] = oz[n].y >= 0 ? py[oz[n].y] : R(0);
#pragma unroll
            for (int n = 0; n < NP; ++n) {
                v[n] += s0[n];
                v[n] += s1[n];
            }
            if (ps.deep) {  // a third and fourth cover, at a ragged mesh's seam
#pragma unroll
                for (int n = 0; n < NP; ++n) {
                    const int z = z0 + 32 * n;
                    if (!near_seam(z, z, Nz) || z >= Nz) continue;
                    const int2 d = __ldg(reinterpret_cast<const int2*>(&zoff[32 * n]) + 1);
                    if (d.x >= 0) v[n] += py[d.x];
                    if (d.y >= 0) v[n] += py[d.y];
                }
            }
        }
    }
}

template <typename R>
__global__ void __launch_bounds__(kFftThreads)
k_fft_z_r2c(Geo g, GenEngine<R> eng, const R* __restrict__ in, typename CT<R>::C* __restrict__ out, int rows, int pairs,
            PatchSrc<R> ps) {
    pdl_enter();
    typedef typename CT<R>::C C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // lines interleaved in shared memory: point t of line p at a[t * pairs + p]
    // (pairs odd, so that a run of t is conflict-free; lanes walk the lines
    // in the FFT stages)
    const int Nz = eng.len(), Hz = g.Hz, PL = pairs;
    C* a = reinterpret_cast<C*>(smem_raw);
    C* b = a + pairs * Nz;
    const int pair0 = blockIdx.x * pairs;
    const int npairs_total = (rows + 1) / 2;
    const int np = min(pairs, npairs_total - pair0);
    if (ps.patch) {
        // a warp folds 32 NP points of a pair's rows at a time
        constexpr int NP = sizeof(R) == 4 ? 4 : 2;
        const int nch = (Nz + 32 * NP - 1) / (32 * NP);
        for (int i = threadIdx.x >> 5; i < np * nch; i += kFftThreads >> 5) {
            const int p = i / nch, z0 = (i - p * nch) * (32 * NP) + (threadIdx.x & 31), r0 = 2 * (pair0 + p);
            R va[NP], vb[NP] = {};
            fold_points<R, NP>(g, ps, r0, z0, Nz, va);
            if (r0 + 1 < rows) fold_points<R, NP>(g, ps, r0 + 1, z0, Nz, vb);
#pragma unroll
            for (int n = 0; n < NP; ++n)
                if (z0 + 32 * n < Nz) a[(z0 + 32 * n) * PL + p] = CT<R>::mk(va[n], vb[n]);
        }
    } else {
        LINE_LOOP(p, t, np, Nz) {
            const int r0 = 2 * (pair0 + p), r1 = r0 + 1;
            const R va = in[(int64_t)r0 * Nz + t];
            const R vb = r1 < rows ? in[(int64_t)r1 * Nz + t] : R(0);
            a[t * PL + p] = CT<R>::mk(va, vb);
        }
    }
    __syncthreads();
    C* res = eng.template run<-1, true>(a, b, np, 1, PL);
    LINE_LOOP(p, k, np, Hz) {
        const int r0 = 2 * (pair0 + p), r1 = r0 + 1;
        const C z = res[k * PL + p];
        const C zc = cconj(res[(k == 0 ? 0 : Nz - k) * PL + p]);
        const C x0 = cscale(cadd(z, zc), R(0.5));
        const C d = csub(z, zc);  // = 2 i X1
        out[(int64_t)r0 * Hz + k] = x0;
        if (r1 < rows) out[(int64_t)r1 * Hz + k] = CT<R>::mk(R(0.5) * d.y, R(-0.5) * d.x);
    }
}

template <typename T>
cudaError_t launch_fft_z_r2c(cudaStream_t s, const Geo& g, const Radix& rz, const typename Cx<T>::t* tw,
                             const T* in, typename Cx<T>::t* out, const PatchSrc<T>& ps) {
    const cudaError_t re = reg_z_r2c<T>(s, g, tw, in, out, ps);
    if (re != cudaErrorNotSupported) return re;
    const int rows = g.N[0] * g.N[1];
    // up to 15 row pairs (an odd count) per block, within 32 KB of shared memory,
    // and no more than give every SM a block (32 x 32 x 243: 38 -> 26 us)
    int pairs = (int)((32 * 1024) / (2 * g.N[2] * sizeof(typename Cx<T>::t)));
    pairs = pairs < 1 ? 1 : (pairs > 15 ? 15 : pairs);
    const int npairs = (rows + 1) / 2, nsm = device_sms();
    pairs = min(pairs, (npairs + nsm - 1) / nsm) | 1;
    const size_t smem = 2ull * pairs * g.N[2] * sizeof(typename Cx<T>::t);
    auto kern = k_fft_z_r2c<T>;
    cudaError_t e = set_smem(kern, smem);
    if (e != cudaSuccess) return e;
    return launch_k(kern, dim3((npairs + pairs - 1) / pairs), dim3(kFftThreads), smem, s, g, GenEngine<T>{rz, tw}, in,
                    out, rows, pairs, ps);
}

// ------------------------------------------------------------------ strided-line C2C
// axis 1: lines along y (outer index x); axis 0: lines along x (outer index y).
// Four resident blocks (64 registers): with the lines per block chosen for it,
// the strided passes run in one round of blocks at the workload sizes.
template <typename R, int SIGN>
__global__ void __launch_bounds__(kFftThreads, 4)
k_fft_bundle(Geo g, int axis, LineBlocks lb, GenEngine<R> eng, typename CT<R>::C* __restrict__ data) {
    pdl_enter();
    typedef typename CT<R>::C C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int Hz = g.Hz, L = eng.len(), B = lb.B;
    const int64_t es = axis == 1 ? (int64_t)Hz : (int64_t)g.N[1] * Hz;  // along the line
    const int64_t os = axis == 1 ? (int64_t)g.N[1] * Hz : (int64_t)Hz;  // between outer rows
    const int64_t nlines = (int64_t)(axis == 1 ? g.N[0] : g.N[1]) * Hz;
    const int64_t f0 = (int64_t)blockIdx.x * B;
    const int nl = (int)min((int64_t)B, nlines - f0);
    const int l = threadIdx.x & 15;  // this thread's line (B <= 16)
    const int64_t fl = f0 + l;
    const int64_t loff = (fl / Hz) * os + fl % Hz;
    C* a = reinterpret_cast<C*>(smem_raw);
    C* b = a + L * B;
    if (l < nl) {
#pragma unroll
        for (int t = threadIdx.x >> 4; t < L; t += kFftThreads >> 4) a[t * B + l] = data[loff + t * es];
    }
    __syncthreads();
    C* res = eng.template run<SIGN, true>(a, b, nl, 1, B);
    if (l < nl) {
#pragma unroll
        for (int t = threadIdx.x >> 4; t < L; t += kFftThreads >> 4) data[loff + t * es] = res[t * B + l];
    }
}

template <typename T>
cudaError_t launch_fft_bundle(cudaStream_t s, const Geo& g, int axis, int sign, const Radix& r, const LineBlocks& lb,
                              const typename Cx<T>::t* tw, typename Cx<T>::t* data) {
    const cudaError_t re = reg_lines<T>(s, g, axis, sign, lb, tw, data);
    if (re != cudaErrorNotSupported) return re;
    const size_t smem = 2ull * r.L * lb.B * sizeof(typename Cx<T>::t);
    auto kern = sign < 0 ? k_fft_bundle<T, -1> : k_fft_bundle<T, 1>;
    cudaError_t e = set_smem(kern, smem);
    if (e != cudaSuccess) return e;
    return launch_k(kern, dim3(lb.nblk), dim3(kFftThreads), smem, s, g, axis, lb, GenEngine<T>{r, tw}, data);
}

// a / b for the virial coefficient: in FP32 the 2-ulp hardware quotient (the
// coefficient enters sums that are accurate to ~1e-7 anyway), in FP64 exact
__device__ __forceinline__ float div_approx(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double div_approx(double a, double b) { return a / b; }

// ------------------------------------------------------------------ x + influence
//
// Per block: B consecutive lines along x, numbered y Hz + kz.
//   1. forward FFT along x  -> rho_hat(k) up to the 1/h^3 factor;
//   2. per mode: G, the energy term e = w G |rho_hat|^2 V/(2 N^2) and the virial
//      terms e (delta_ab - 2 (1 + k^2/(4 beta^2)) k_a k_b / k^2), summed plainly
//      over a thread's Nx/16 modes (a relative error of at most Nx/16 roundings
//      of that short sum), then reduced across threads and blocks with
//      compensated (TwoSum) pairs;
//   3. P = G rho_hat / (N h^3) and -i kx' P (kx' = 0 on the Nyquist index);
//   4. inverse FFT along x of both; P -> S (in place), -i kx' P -> Bx.
// A block of the y inverse sums the per-block partials (TwoSum in the mesh
// precision, hi + lo in FP64 at the end) in a fixed order.
//
// Half-spectrum weights: w = 1 on the kz = 0 plane (and kz = Nz/2 for even Nz),
// 2 elsewhere, standing for the mirror mode -k.  For the off-diagonal virial a
// mirrored mode whose x (or y) index is the Nyquist index keeps that component's
// sign (the index maps to itself, m = +N/2), so a product k_a k_b survives the
// pairing only when both or neither of its components flip sign.
template <typename R>
__global__ void __launch_bounds__(kFftThreads, 4)
k_fft_x_influence(Geo g, LineBlocks lb, GenEngine<R> eng, const R* __restrict__ G, R beta, R e_scale, R c_field,
                  typename CT<R>::C* __restrict__ S, typename CT<R>::C* __restrict__ Bx, R* __restrict__ partial) {
    pdl_enter();
    typedef typename CT<R>::C C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ R red[kFftThreads / 32][14];
    const int Nx = eng.len(), Ny = g.N[1], Nz = g.N[2], Hz = g.Hz, B = lb.B;
    // lines along x, numbered f = y Hz + kz: a block's B lines are consecutive in memory
    const int64_t es = (int64_t)Ny * Hz;
    const int64_t f0 = (int64_t)blockIdx.x * B;
    const int nl = (int)min((int64_t)B, es - f0);
    const int lt = threadIdx.x & 15;  // this thread's line (B <= 16)
    const int yl = (int)((f0 + lt) / Hz), kzl = (int)((f0 + lt) - (int64_t)yl * Hz);
    // three line buffers; each transform returns the one holding its result
    // and the others are reused as they free up
    C* a0 = reinterpret_cast<C*>(smem_raw);
    C* a1 = a0 + Nx * B;
    C* b0 = a1 + Nx * B;
    C* base = S + f0;
    BUNDLE_LOOP(t, l, Nx, nl) a0[t * B + l] = base[t * es + l];
    __syncthreads();
    C* rh = eng.template run<-1, true>(a0, a1, nl, 1, B);
    C* pbuf = (rh == a0) ? a1 : a0;  // free partner of the result buffer

    const int my = yl <= Ny / 2 ? yl : yl - Ny;
    const R ky = kfac<R>(g, 1) * my;
    const bool nyq_y = (Ny % 2 == 0) && (yl == Ny / 2);
    const R inv4b2 = R(1) / (R(4) * beta * beta);
    R acc[7];
#pragma unroll
    for (int q = 0; q < 7; ++q) acc[q] = R(0);
    const int kz = kzl;
    const R kzv = kfac<R>(g, 2) * kz;
    const bool plane1 = (kz == 0) || ((Nz % 2 == 0) && (kz == Nz / 2));
    const R w = plane1 ? R(1) : R(2);
    auto mode = [&](int t, R gk) {  // mode (t, line lt): energy and virial terms, P and -i kx' P
        const int mx = t <= Nx / 2 ? t : t - Nx;
        const R kx = kfac<R>(g, 0) * mx;
        const bool nyq_x = (Nx % 2 == 0) && (t == Nx / 2);
        const C v = rh[t * B + lt];
        const R k2 = kx * kx + ky * ky + kzv * kzv;
        if (k2 > R(0)) {
            const R e = w * e_scale * gk * (v.x * v.x + v.y * v.y);
            const R c = div_approx(R(2) * (R(1) + k2 * inv4b2), k2);
            const R fxy = (plane1 || (nyq_x == nyq_y)) ? R(1) : R(0);
            const R fxz = (plane1 || !nyq_x) ? R(1) : R(0);
            const R fyz = (plane1 || !nyq_y) ? R(1) : R(0);
            acc[0] += e;
            acc[1] += e * (R(1) - c * kx * kx);
            acc[2] += e * (R(1) - c * ky * ky);
            acc[3] += e * (R(1) - c * kzv * kzv);
            acc[4] -= e * c * kx * ky * fxy;
            acc[5] -= e * c * kx * kzv * fxz;
            acc[6] -= e * c * ky * kzv * fyz;
        }
        const C P = cscale(v, gk * c_field);
        const R kxd = nyq_x ? R(0) : kx;
        pbuf[t * B + lt] = P;
        b0[t * B + lt] = CT<R>::mk(kxd * P.y, -kxd * P.x);  // -i kx' P
    };
    if (lt < nl) {
#pragma unroll 1
        for (int t = threadIdx.x >> 4; t < Nx; t += kFftThreads >> 4) mode(t, G[(int64_t)t * es + f0 + lt]);
    }
    __syncthreads();
    C* rA = eng.template run<1, true>(pbuf, rh, nl, 1, B);  // rho_hat is no longer needed: scratch
    C* fr = (rA == pbuf) ? rh : pbuf;
    C* rB = eng.template run<1, true>(b0, fr, nl, 1, B);
    C* obx = Bx + f0;
    BUNDLE_LOOP(t, l, Nx, nl) {
        base[t * es + l] = rA[t * B + l];
        obx[t * es + l] = rB[t * B + l];
    }

    // block reduction of the 7 compensated sums: (hi, lo) pairs combined with TwoSum
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < 7; ++q) {
        R h = acc[q], lo = R(0);
        for (int off = 16; off > 0; off >>= 1) {
            const R h2 = __shfl_down_sync(0xffffffffu, h, off);
            const R l2 = __shfl_down_sync(0xffffffffu, lo, off);
            two_sum_pair(h, lo, h2, l2);
        }
        if (lane == 0) { red[warp][2 * q] = h; red[warp][2 * q + 1] = lo; }
    }
    __syncthreads();
    if (threadIdx.x < 7) {
        const int q = threadIdx.x;
        R h = red[0][2 * q], lo = red[0][2 * q + 1];
        for (int w = 1; w < kFftThreads / 32; ++w) two_sum_pair(h, lo, red[w][2 * q], red[w][2 * q + 1]);
        partial[(int64_t)blockIdx.x * 14 + 2 * q] = h;
        partial[(int64_t)blockIdx.x * 14 + 2 * q + 1] = lo;
    }
}

int x_influence_blocks(const LineBlocks& lb) { return lb.nblk; }

template <typename T>
cudaError_t launch_fft_x_influence(cudaStream_t s, const Geo& g, const Radix& rx, const LineBlocks& lb,
                                   const typename Cx<T>::t* tw, const T* G, double beta, double e_scale,
                                   double c_field, typename Cx<T>::t* S, typename Cx<T>::t* Bx, T* partial) {
    const cudaError_t re = reg_x_influence<T>(s, g, lb, tw, G, beta, e_scale, c_field, S, Bx, partial);
    if (re != cudaErrorNotSupported) return re;
    const size_t smem = 3ull * g.N[0] * lb.B * sizeof(typename Cx<T>::t);
    auto kern = k_fft_x_influence<T>;
    cudaError_t e = set_smem(kern, smem);
    if (e != cudaSuccess) return e;
    return launch_k(kern, dim3(x_influence_blocks(lb)), dim3(kFftThreads), smem, s, g, lb, GenEngine<T>{rx, tw}, G,
                    (T)beta, (T)e_scale, (T)c_field, S, Bx, partial);
}

// ------------------------------------------------------------------ y inverse, three outputs
// C = IFFT_y(A), D = IFFT_y(-i ky' A), Ex' = IFFT_y(Bx); C overwrites A, Ex'
// overwrites Bx.  Block 0 sums the x pass's energy partials beside the others.
template <typename R>
__global__ void __launch_bounds__(kFftThreads, 4)
k_fft_y_inverse3(Geo g, LineBlocks lb, GenEngine<R> eng, typename CT<R>::C* __restrict__ A, typename CT<R>::C* __restrict__ Bx,
                 typename CT<R>::C* __restrict__ D, const R* __restrict__ partial, int npart, double prefactor,
                 double* __restrict__ energy, double* __restrict__ virial) {
    pdl_enter();
    if (blockIdx.x == 0) {
        finish_energy(partial, npart, prefactor, energy, virial);
        return;
    }
    typedef typename CT<R>::C C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int Ny = eng.len(), Hz = g.Hz, B = lb.B;
    // lines along y, numbered f = x Hz + kz; line f starts at x Ny Hz + kz
    const int64_t f0 = (int64_t)(blockIdx.x - 1) * B;
    const int nl = (int)min((int64_t)B, (int64_t)g.N[0] * Hz - f0);
    const int64_t fl = f0 + (threadIdx.x & 15);  // this thread's line (B <= 16)
    const int64_t loff = (fl / Hz) * ((int64_t)Ny * Hz) + fl % Hz;
    // four line buffers: the three inputs and a scratch that rotates, each
    // transform leaving its result in one of the two it used
    const int sz = Ny * B;
    C* p0 = reinterpret_cast<C*>(smem_raw);
    C* p1 = p0 + sz;
    C* p2 = p1 + sz;
    C* scr = p2 + sz;
    BUNDLE_LOOP(t, l, Ny, nl) {
        const C va = A[loff + (int64_t)t * Hz];
        const int my = t <= Ny / 2 ? t : t - Ny;
        const R kyd = ((Ny % 2 == 0) && (t == Ny / 2)) ? R(0) : kfac<R>(g, 1) * my;
        p0[t * B + l] = va;
        p1[t * B + l] = CT<R>::mk(kyd * va.y, -kyd * va.x);
        p2[t * B + l] = Bx[loff + (int64_t)t * Hz];
    }
    __syncthreads();
    C* rC = eng.template run<1, true>(p0, scr, nl, 1, B);
    if (rC == scr) scr = p0;
    C* rD = eng.template run<1, true>(p1, scr, nl, 1, B);
    if (rD == scr) scr = p1;
    C* rE = eng.template run<1, true>(p2, scr, nl, 1, B);
    BUNDLE_LOOP(t, l, Ny, nl) {
        A[loff + (int64_t)t * Hz] = rC[t * B + l];
        D[loff + (int64_t)t * Hz] = rD[t * B + l];
        Bx[loff + (int64_t)t * Hz] = rE[t * B + l];
    }
}

template <typename T>
cudaError_t launch_fft_y_inverse3(cudaStream_t s, const Geo& g, const Radix& ry, const LineBlocks& lb,
                                  const typename Cx<T>::t* tw, typename Cx<T>::t* A, typename Cx<T>::t* Bx,
                                  typename Cx<T>::t* D, const T* partial, int npart, double prefactor,
                                  double* energy, double* virial) {
    const cudaError_t re = reg_y_inverse3<T>(s, g, lb, tw, A, Bx, D, partial, npart, prefactor, energy, virial);
    if (re != cudaErrorNotSupported) return re;
    const size_t smem = 4ull * g.N[1] * lb.B * sizeof(typename Cx<T>::t);
    auto kern = k_fft_y_inverse3<T>;
    cudaError_t e = set_smem(kern, smem);
    if (e != cudaSuccess) return e;
    return launch_k(kern, dim3(lb.nblk + 1), dim3(kFftThreads), smem, s, g, lb, GenEngine<T>{ry, tw}, A, Bx, D,
                    partial, npart, prefactor, energy, virial);
}

// ------------------------------------------------------------------ z inverse (C2R)
template <typename R>
__global__ void __launch_bounds__(kFftThreads, 6)  // six resident blocks: two rounds instead of three
k_fft_z_c2r(Geo g, GenEngine<R> eng, ZOut zo, int rows, int pairs) {
    pdl_enter();
    typedef typename CT<R>::C C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // lines interleaved in shared memory: point t of line L at a[t * PL + L],
    // PL odd (a run of t is conflict-free); lanes walk the lines in the stages
    const int Nz = eng.len(), Hz = g.Hz;
    const int nf = zo.nf;
    const int PL = (nf * pairs) | 1;
    C* a = reinterpret_cast<C*>(smem_raw);
    C* b = a + PL * Nz;
    const int pair0 = blockIdx.x * pairs;
    const int npairs_total = (rows + 1) / 2;
    const int np = min(pairs, npairs_total - pair0);
    const int nlines = nf * np;
    const bool even = (Nz % 2) == 0;
    LINE_LOOP(line, t, nlines, Nz) {
        const int f = line / np, p = line - f * np;
        const int r0 = 2 * (pair0 + p), r1 = r0 + 1;
        const C* src = reinterpret_cast<const C*>(pick4(zo.src, f));
        const int mulkz = pick4(zo.mulkz, f);
        // Hermitian extension: t < Hz reads the half row, t >= Hz the conjugate of Nz - t
        const int kk = t < Hz ? t : Nz - t;
        const bool cj = t >= Hz;
        const bool realonly = (kk == 0) || (even && kk == Nz / 2);
        R kzd = R(0);
        if (mulkz && !(even && kk == Nz / 2)) kzd = kfac<R>(g, 2) * kk;
        C h0 = src[(int64_t)r0 * Hz + kk];
        C h1 = r1 < rows ? src[(int64_t)r1 * Hz + kk] : CT<R>::mk(R(0), R(0));
        if (mulkz) {  // -i kz' h
            h0 = CT<R>::mk(kzd * h0.y, -kzd * h0.x);
            h1 = CT<R>::mk(kzd * h1.y, -kzd * h1.x);
        }
        if (realonly) { h0.y = R(0); h1.y = R(0); }
        if (cj) { h0.y = -h0.y; h1.y = -h1.y; }
        a[t * PL + line] = CT<R>::mk(h0.x - h1.y, h0.y + h1.x);  // h0 + i h1
    }
    __syncthreads();
    C* res = eng.template run<1, true>(a, b, nlines, 1, PL);
    if (!zo.fl.padded) {
        LINE_LOOP(line, t, nlines, Nz) {
            const int f = line / np, p = line - f * np;
            const int r0 = 2 * (pair0 + p), r1 = r0 + 1;
            R* out = reinterpret_cast<R*>(pick4(zo.out, f));
            const C z = res[t * PL + line];
            out[(int64_t)r0 * Nz + t] = z.x;
            if (r1 < rows) out[(int64_t)r1 * Nz + t] = z.y;
        }
        return;
    }
    // padded: the fields of a point are interleaved (E_x, E_y, E_z, 0) and
    // stored with one vector store, the potential (a fourth output) goes to
    // its own padded mesh; every output row also lands on its
    // periodic ghost images, and each row is extended by p - 1 ghost points
    // along z.  One warp per output row, lanes along z.
    const FieldLayout& fl = zo.fl;
    const int Ny = g.N[1], kmin = g.kmin;
    const int zlen = Nz + g.order - 1;
    typedef typename CT<R>::C4 V4;
    V4* out = reinterpret_cast<V4*>(zo.out[0]);
    R* phi = nf == 4 ? reinterpret_cast<R*>(zo.out[3]) : nullptr;  // padded potential, one value a point
    for (int pr = threadIdx.x >> 5; pr < 2 * np; pr += kFftThreads >> 5) {
        const int p = pr >> 1, half = pr & 1;
        const int r = 2 * (pair0 + p) + half;
        if (r >= rows) continue;
        const int x = r / Ny, y = r - x * Ny;
        const int px0 = x - kmin, py0 = y - kmin;
        // at most one ghost image per axis (Xp < 2 Nx)
        const int Nx = g.N[0];
        const int pxg = px0 + Nx < fl.Xp ? px0 + Nx : (px0 - Nx >= 0 ? px0 - Nx : -1);
        const int pyg = py0 + Ny < fl.Yp ? py0 + Ny : (py0 - Ny >= 0 ? py0 - Ny : -1);
        const int64_t r00 = ((int64_t)px0 * fl.Yp + py0) * fl.Zp;  // first point of each image row
        const int64_t r10 = pxg >= 0 ? ((int64_t)pxg * fl.Yp + py0) * fl.Zp : -1;
        const int64_t r01 = pyg >= 0 ? ((int64_t)px0 * fl.Yp + pyg) * fl.Zp : -1;
        const int64_t r11 = (pxg >= 0 && pyg >= 0) ? ((int64_t)pxg * fl.Yp + pyg) * fl.Zp : -1;
        for (int pz = threadIdx.x & 31; pz < zlen; pz += 32) {
            int zz = pz + kmin;
            zz += zz < 0 ? Nz : 0;
            zz -= zz >= Nz ? Nz : 0;
            const C* rz = res + zz * PL + p;  // field f of this pair at rz[f * np]
            R v[4];
#pragma unroll
            for (int f = 0; f < 4; ++f) {
                const C zv = f < nf ? rz[f * np] : CT<R>::mk(R(0), R(0));
                v[f] = half ? zv.y : zv.x;
            }
            const V4 w = CT<R>::mk4(v[0], v[1], v[2], R(0));
            out[r00 + pz] = w;
            if (r10 >= 0) out[r10 + pz] = w;
            if (r01 >= 0) out[r01 + pz] = w;
            if (r11 >= 0) out[r11 + pz] = w;
            if (phi) {
                phi[r00 + pz] = v[3];
                if (r10 >= 0) phi[r10 + pz] = v[3];
                if (r01 >= 0) phi[r01 + pz] = v[3];
                if (r11 >= 0) phi[r11 + pz] = v[3];
            }
        }
    }
}

template <typename T>
cudaError_t launch_fft_z_c2r(cudaStream_t s, const Geo& g, const Radix& rz, const typename Cx<T>::t* tw, int nf,
                             const typename Cx<T>::t* const* src, const int* mulkz, T* const* out,
                             const FieldLayout& fl) {
    ZOut zo;
    zo.nf = nf;
    zo.fl = fl;
    for (int f = 0; f < 4; ++f) {
        zo.src[f] = f < nf ? src[f] : nullptr;
        zo.out[f] = f < nf ? out[f] : nullptr;
        zo.mulkz[f] = f < nf ? mulkz[f] : 0;
    }
    const cudaError_t re = reg_z_c2r<T>(s, g, tw, zo);
    if (re != cudaErrorNotSupported) return re;
    const int rows = g.N[0] * g.N[1];
    // at most 16 lines (nf fields x pairs) per block, the 16 lanes of a group
    // each taking one line in the FFT stages
    int pairs = 16 / nf;
    if (pairs < 1) pairs = 1;
    const int npairs = (rows + 1) / 2;
    const size_t smem = 2ull * ((nf * pairs) | 1) * g.N[2] * sizeof(typename Cx<T>::t);
    auto kern = k_fft_z_c2r<T>;
    cudaError_t e = set_smem(kern, smem);
    if (e != cudaSuccess) return e;
    return launch_k(kern, dim3((npairs + pairs - 1) / pairs), dim3(kFftThreads), smem, s, g, GenEngine<T>{rz, tw}, zo,
                    rows, pairs);
}

// B for one pass: the fewest rounds of resident blocks, then the fewest
// blocks on the busiest SM (a block costs about the same for any B <= 16:
// its lanes are laid out for 16 lines), then the larger B.  resident(B) gives
// the resident blocks per SM.
template <typename F>
static LineBlocks pick_line_blocks(F resident, int maxB, int64_t lines, int nsm) {
    LineBlocks best{1, (int)lines};
    int64_t best_rounds = -1, best_busy = 0;
    for (int B = 1; B <= maxB; ++B) {
        const int per = resident(B);
        if (per < 1) continue;
        const int64_t blocks = (lines + B - 1) / B;
        const int64_t rounds = (blocks + (int64_t)per * nsm - 1) / ((int64_t)per * nsm);
        const int64_t busy = (blocks + nsm - 1) / nsm;
        if (best_rounds < 0 || rounds < best_rounds || (rounds == best_rounds && busy <= best_busy)) {
            best_rounds = rounds;
            best_busy = busy;
            best = LineBlocks{B, (int)blocks};
        }
    }
    return best;
}

template <typename T, typename K>
static LineBlocks pass_line_blocks(int pass, K kern, int nbuf, int L, int64_t lines, int nsm) {
    const int reg = reg_resident<T>(pass, L);
    if (reg > 0) return pick_line_blocks([&](int) { return reg; }, 16, lines, nsm);
    const size_t per_line = nbuf * sizeof(typename Cx<T>::t) * L;
    int maxB = 16;
    while (maxB > 1 && per_line * maxB > 227 * 1024) --maxB;
    if (set_smem(kern, per_line * maxB) != cudaSuccess) {
        cudaGetLastError();
        return LineBlocks{1, (int)lines};
    }
    return pick_line_blocks(
        [&](int B) {
            int per = 0;
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, kFftThreads, per_line * B) != cudaSuccess) {
                cudaGetLastError();
                return 0;
            }
            return per;
        },
        maxB, lines, nsm);
}

template <typename T>
cudaError_t choose_line_blocks(const Geo& g, const Radix rad[3], int nsm, LineBlocks lb[4]) {
    const int64_t Hz = g.Hz;
    const int Lx = rad[0].L, Ly = rad[1].L;
    lb[LB_Y] = pass_line_blocks<T>(LB_Y, k_fft_bundle<T, -1>, 2, Ly, g.N[0] * Hz, nsm);
    lb[LB_Y_INVERSE3] = pass_line_blocks<T>(LB_Y_INVERSE3, k_fft_y_inverse3<T>, 4, Ly, g.N[0] * Hz, nsm);
    lb[LB_X_INFLUENCE] = pass_line_blocks<T>(LB_X_INFLUENCE, k_fft_x_influence<T>, 3, Lx, g.N[1] * Hz, nsm);
    lb[LB_X] = pass_line_blocks<T>(LB_X, k_fft_bundle<T, 1>, 2, Lx, g.N[1] * Hz, nsm);
    return cudaSuccess;
}

#define PPPM_INST_FFT(T)                                                                                           \
    template cudaError_t launch_fft_z_r2c<T>(cudaStream_t, const Geo&, const Radix&, const Cx<T>::t*, const T*,    \
                                             Cx<T>::t*, const PatchSrc<T>&);                                       \
    template cudaError_t choose_line_blocks<T>(const Geo&, const Radix*, int, LineBlocks*);                      \
    template cudaError_t launch_fft_bundle<T>(cudaStream_t, const Geo&, int, int, const Radix&, const LineBlocks&, \
                                              const Cx<T>::t*, Cx<T>::t*);                                         \
    template cudaError_t launch_fft_x_influence<T>(cudaStream_t, const Geo&, const Radix&, const LineBlocks&,      \
                                                   const Cx<T>::t*, const T*, double, double, double, Cx<T>::t*,   \
                                                   Cx<T>::t*, T*);                                                 \
    template cudaError_t launch_fft_y_inverse3<T>(cudaStream_t, const Geo&, const Radix&, const LineBlocks&,       \
                                                  const Cx<T>::t*, Cx<T>::t*, Cx<T>::t*, Cx<T>::t*, const T*, int, \
                                                  double, double*, double*);                                       \
    template cudaError_t launch_fft_z_c2r<T>(cudaStream_t, const Geo&, const Radix&, const Cx<T>::t*, int,         \
                                             const Cx<T>::t* const*, const int*, T* const*, const FieldLayout&);
PPPM_INST_FFT(float)
PPPM_INST_FFT(double)

}  // namespace pppm
