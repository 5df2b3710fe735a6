// Fold of the Wannier-centroid forces onto atoms, Eq. DPLR:F_final.
//
// W_n = R_host(n) + Delta_n(R) (Eq. DPLR:Wn), so the long-range force on atom j
// is its own site force, plus the force on every WC it hosts, plus
// J^T F_W(n) for every Jacobian block J = dDelta_n/dR_j listed in its row.
// Every sum has a fixed order: the result is bitwise reproducible.
//
// The kernels stream the blocks once (40 bytes each in FP32, 76 in FP64) and read
// a WC force for each (12 or 24 bytes, scattered over a table that L2 holds).
// Bound by the latency of those reads and the instructions between them: the
// stream alone takes 34 us of the 68 for 216,576 atoms with up to 27 blocks each
// (72,192 molecules, FP32).  So a lane fetches the indices of its next blocks
// while it works on the current ones, and reads a force as one or two 16-byte
// vectors (three loads of one value each look up their cache line three times).
//
// The two precisions split the work differently.  In FP32 (k_wc_fold_lanes) the
// lanes of a warp take consecutive blocks, add each to its row's accumulator,
// and sum four rows at once with a transposing butterfly: 90.4 -> 67.8 us against
// four xor butterflies and indices fetched when needed; 200,000 atoms of 27 blocks
// 86.5 -> 65.8, of 4 blocks 28.9 -> 22.9, 100,000 of 0-54 43.7 -> 38.9 (16,000 of 200
// blocks 33.9 -> 35.0: the one shape that lost).  Blocks staged through
// shared memory took 69-92 us (fewer resident warps).  In FP64, whose additions
// are a 64th as fast, every accumulator that a block is masked into costs
// (27 blocks, 100,000 atoms: 327 us), so a row belongs to a set of lanes
// (k_wc_fold_rows, 98.6 us), which read its blocks from shared memory.
#include <climits>
#include <cstdint>

#include "internal.cuh"

namespace pppm {

constexpr int kFoldWarps = 4;
constexpr int kCount = 1 << 20;  // blocks of a group that are counted in 32 bits (FP32)
constexpr int kLaneBlocks = 7, kRowBlocks = 5;  // resident blocks an SM: registers (FP32), the stages (FP64)

struct FoldStage {
    static constexpr int CAP = 128;  // blocks
    // the blocks, with the bytes before the first one in its 16-byte vector (and
    // room for the bytes after the last one in its own)
    __align__(16) unsigned char jac[CAP * 9 * sizeof(double) + 32];
};

template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst, const void* src) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(BYTES) : "memory");
}

// Starts the copy of `bytes` bytes of doubles (at most MAX) at src to the place in
// dst with the same offset in a 16-byte vector (returned): whole vectors, value
// by value only where a vector reaches out of the array [base, end).
template <int MAX>
__device__ __forceinline__ int copy_vectors(unsigned char* dst, const char* src, int bytes, const char* base,
                                            const char* end, int lane) {
    const int lead = (int)(reinterpret_cast<uintptr_t>(src) & 15);
    src += 16 * lane - lead;
    dst += 16 * lane;
    bytes += lead - 16 * lane;  // left from this lane's first vector on
    if (src >= base && src + ((bytes + 15) & ~15) <= end) {
#pragma unroll
        for (int o = 0; o < MAX + 16; o += 512)
            if (o < bytes) cp_async<16>(dst + o, src + o);
    } else {
        const int first = lane == 0 ? lead : 0;
        for (int o = 0; o < bytes; o += 512)
            for (int v = o; v < o + 16; v += 8)
                if (v >= first && v < bytes) cp_async<8>(dst + v, src + v);
    }
    return lead;
}

// The three components at p (a row of the forces), which is followed by at
// least one more row: the one or two 16-byte vectors that hold them (one
// request each, where three separate loads fetch their sector three times).
__device__ __forceinline__ void load_row3(const float* p, float& a, float& b, float& c) {
    const uintptr_t at = reinterpret_cast<uintptr_t>(p);
    const float4* v = reinterpret_cast<const float4*>(at & ~uintptr_t(15));
    const bool two = (at & 8) != 0, one = (at & 4) != 0;
    float4 q = *v;
    if (two) {
        const float2 r = *reinterpret_cast<const float2*>(v + 1);
        q = make_float4(q.z, q.w, r.x, r.y);
    }
    a = one ? q.y : q.x;
    b = one ? q.z : q.y;
    c = one ? q.w : q.z;
}
__device__ __forceinline__ void load_row3(const double* p, double& a, double& b, double& c) {
    const uintptr_t at = reinterpret_cast<uintptr_t>(p);
    const double2* v = reinterpret_cast<const double2*>(at & ~uintptr_t(15));
    const bool one = (at & 8) != 0;
    const double2 q = v[0], r = v[1];
    a = one ? q.y : q.x;
    b = one ? r.x : q.y;
    c = one ? r.y : r.x;
}

// FP32: a warp takes groups of R atoms, whose rows are one contiguous run of blocks.
__global__ void __launch_bounds__(kFoldWarps * 32, kLaneBlocks)
k_wc_fold_lanes(int64_t n_atoms, int64_t n_wc, const float* __restrict__ f_sites, const int* __restrict__ host_ptr,
                const int* __restrict__ host_wc, const int64_t* __restrict__ jac_ptr, const int* __restrict__ jac_wc,
                const float* __restrict__ jac, float* __restrict__ f_atoms, int* __restrict__ status) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * kFoldWarps;
    // four atoms share the butterfly (27 blocks a row: four 68 us, one or two
    // more); fewer where their rows are long, or where the last of the warps'
    // turns would be mostly empty (200 blocks a row, 16,000 atoms: 43 us with
    // four, 37 with one)
    int R = n_atoms < 4 * warps ? 1 : n_atoms < 8 * warps ? 2 : 4;
    if (R > 1 && jac_ptr) {
        const int64_t nnz = jac_ptr[n_atoms] - jac_ptr[0];
        R = nnz >= 96 * n_atoms ? 1 : nnz >= 48 * n_atoms ? 2 : R;
    }
    const int64_t groups = (n_atoms + R - 1) / R;
    const float* fw = f_sites + 3 * n_atoms;
    const unsigned nwc = (unsigned)min(n_wc, (int64_t)INT_MAX);
    bool bad = false;
    // lane i: where row i of a group starts (its end from i = R on)
    auto row_ptr = [&](int64_t grp) -> int64_t {
        if (!jac_ptr || grp >= groups) return 0;
        return jac_ptr[min(R * grp + min(lane, R), n_atoms)];
    };
    // a group's first block (k) and blocks (n, those up to kCount)
    auto extent = [&](int64_t ptr, int64_t& k, int& n) {
        k = __shfl_sync(0xffffffffu, ptr, 0);
        n = (int)min(__shfl_sync(0xffffffffu, ptr, 4) - k, (int64_t)kCount);
    };
    // the WC of block i of the n from k on (-1: none)
    auto load_wc = [&](int64_t k, int i, int n) { return i < n ? __ldg(jac_wc + k + i) : -1; };
    int64_t grp = (int64_t)blockIdx.x * kFoldWarps + (threadIdx.x >> 5);
    int64_t ptr = row_ptr(grp), nptr = row_ptr(grp + warps), k;
    int n;
    extent(ptr, k, n);
    int w = load_wc(k, lane, n);
    for (; grp < groups; grp += warps) {
        const int64_t nnptr = row_ptr(grp + 2 * warps);
        // lane 4 r + c: component c of atom R grp + r, its own force and
        // hosted-WC range, which arrive while the rows are summed
        const int64_t j = R * grp + ((lane & 15) >> 2);
        const int comp = lane & 3;
        const bool mine = lane < 4 * R && comp < 3 && j < n_atoms;
        float own = 0.f;
        int h0 = 0, h1 = 0;
        if (mine) {
            own = f_sites[3 * j + comp];
            if (host_ptr) {
                h0 = host_ptr[j];
                h1 = host_ptr[j + 1];
            }
        }
        int64_t nk;
        int nn;
        extent(nptr, nk, nn);
        // where the rows 1, 2, 3 start, in blocks from k on
        int b[3];
#pragma unroll
        for (int r = 0; r < 3; ++r)
            b[r] = (int)min(max(__shfl_sync(0xffffffffu, ptr, r + 1) - k, (int64_t)0), (int64_t)kCount);
        float acc[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) acc[i] = 0.f;
        for (int i = lane;;) {
            float v[9], g[3] = {0.f, 0.f, 0.f};
            const bool in = (unsigned)w < nwc;
            bad |= !in && i < n;
#pragma unroll
            for (int e = 0; e < 9; ++e) v[e] = 0.f;
            if (in) {
                const float* f = fw + 3 * (int64_t)w;
                if ((unsigned)w + 1 < nwc) {
                    load_row3(f, g[0], g[1], g[2]);
                } else {
                    g[0] = f[0];
                    g[1] = f[1];
                    g[2] = f[2];
                }
                const float* J = jac + 9 * (k + i);
#pragma unroll
                for (int e = 0; e < 9; ++e) v[e] = __ldg(J + e);
            }
            const int row = (i >= b[0]) + (i >= b[1]) + (i >= b[2]);
            const bool last = n - (i - lane) <= 32;  // uniform
            i += 32;
            w = last ? load_wc(nk, lane, nn) : load_wc(k, i, n);
            // (J^T g)_b = sum_a J[a][b] g_a
            float c[3];
#pragma unroll
            for (int d = 0; d < 3; ++d) c[d] = v[d] * g[0] + v[3 + d] * g[1] + v[6 + d] * g[2];
#pragma unroll
            for (int r = 0; r < 4; ++r)
                if (row == r) {
                    acc[4 * r] += c[0];
                    acc[4 * r + 1] += c[1];
                    acc[4 * r + 2] += c[2];
                }
            if (last) break;
        }
        if (n == kCount) {  // the group's further blocks, counted in 64 bits
            const int64_t end = __shfl_sync(0xffffffffu, ptr, 4);
            const int64_t p1 = __shfl_sync(0xffffffffu, ptr, 1), p2 = __shfl_sync(0xffffffffu, ptr, 2),
                          p3 = __shfl_sync(0xffffffffu, ptr, 3);
#pragma unroll 1
            for (int64_t q = k + n + lane; q < end; q += 32) {
                const int m = jac_wc[q];
                if ((unsigned)m >= nwc) {
                    bad = true;
                    continue;
                }
                const float *f = fw + 3 * (int64_t)m, *J = jac + 9 * q;
                const int row = (q >= p1) + (q >= p2) + (q >= p3);
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    const float c = J[d] * f[0] + J[3 + d] * f[1] + J[6 + d] * f[2];
#pragma unroll
                    for (int r = 0; r < 4; ++r) acc[4 * r + d] += row == r ? c : 0.f;
                }
            }
        }
        // sum over the lanes: component c of row r ends in lanes 4 r + c (+ 16)
#pragma unroll
        for (int h = 8; h >= 1; h >>= 1) {
            const bool up = (lane & h) != 0;
#pragma unroll
            for (int i = 0; i < h; ++i) {
                if (h >= 4 && (i & 3) == 3) continue;  // no component 3
                const float send = up ? acc[i] : acc[i + h];
                const float keep = up ? acc[i + h] : acc[i];
                acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, h);
            }
        }
        acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 16);
        if (mine) {
            for (int h = h0; h < h1; ++h) {
                const int m = host_wc[h];
                if ((unsigned)m < nwc) own += fw[3 * (int64_t)m + comp];
                else bad = true;
            }
            f_atoms[3 * j + comp] = own + acc[0];
        }
        ptr = nptr;
        nptr = nnptr;
        k = nk;
        n = nn;
    }
    if (bad && status) atomicOr(status, 1);
}

// FP64: a warp takes runs of up to 32 atoms, 32 / rows lanes a row, and streams
// their blocks through its stage in whole 16-byte vectors (cp.async), a piece of
// up to CAP blocks at a time.
__global__ void __launch_bounds__(kFoldWarps * 32, kRowBlocks)
k_wc_fold_rows(int64_t n_atoms, int64_t n_wc, const double* __restrict__ f_sites, const int* __restrict__ host_ptr,
               const int* __restrict__ host_wc, const int64_t* __restrict__ jac_ptr, const int* __restrict__ jac_wc,
               const double* __restrict__ jac, double* __restrict__ f_atoms, int* __restrict__ status) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    typedef double T;
    constexpr int CAP = FoldStage::CAP, BLOCK = 9 * (int)sizeof(T);  // bytes a block
    FoldStage& S = reinterpret_cast<FoldStage*>(smem_raw)[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * kFoldWarps;
    const T* fw = f_sites + 3 * n_atoms;
    // rows of a run, 32 at most: about 7/8 of the stage on average, and few
    // enough that every warp has one
    const int64_t kend = jac_ptr ? jac_ptr[n_atoms] : 0, nnz = jac_ptr ? kend - jac_ptr[0] : 0;
    int lg = 0;  // log2 of the lanes of a row
    while (lg < 5 && ((nnz << (5 - lg)) > CAP * 7 / 8 * n_atoms || n_atoms < (warps << (5 - lg)))) ++lg;
    const int G = 1 << lg, rows = 32 >> lg, row = lane >> lg, sub = lane & (G - 1);
    const char* jb = reinterpret_cast<const char*>(jac);
    const char* je = jb + kend * BLOCK;
    const unsigned nwc = (unsigned)min(n_wc, (int64_t)INT_MAX);
    constexpr int U = 2;  // blocks of a lane at a time
    bool bad = false;
    // this lane's row of the run that starts at atom j0
    auto row_range = [&](int64_t j0, int64_t& lo, int64_t& hi) {
        lo = hi = 0;
        if (!jac_ptr || j0 >= n_atoms) return;
        lo = jac_ptr[min(j0 + row, n_atoms)];
        hi = jac_ptr[min(j0 + row + 1, n_atoms)];
    };
    // a piece: up to CAP blocks from k on; this lane's row holds blocks b .. b + n - 1 of it
    struct Piece {
        int64_t k, e;
        int b, n;
    };
    auto piece = [&](int64_t k, int64_t ke, int64_t lo, int64_t hi) {
        Piece p;
        p.k = k;
        p.e = min(k + CAP, ke);
        p.b = (int)(min(max(lo, k), p.e) - k);
        p.n = (int)(min(max(hi, k), p.e) - k) - p.b;
        return p;
    };
    // the WCs of this lane's blocks i0, i0 + G, ... of its row in a piece
    auto load_wc = [&](const Piece& p, int i0, int (&w)[U]) {
        const int* at = jac_wc + p.k + p.b;
#pragma unroll
        for (int u = 0; u < U; ++u) w[u] = i0 + u * G < p.n ? __ldg(at + i0 + u * G) : -1;
    };
    int64_t j0 = ((int64_t)blockIdx.x * kFoldWarps + (threadIdx.x >> 5)) * rows;
    const int64_t step = warps * rows;
    int64_t lo, hi, nlo, nhi;
    row_range(j0, lo, hi);
    row_range(j0 + step, nlo, nhi);
    int64_t ke = __shfl_sync(0xffffffffu, hi, 31);
    Piece p = piece(__shfl_sync(0xffffffffu, lo, 0), ke, lo, hi);
    int w[U];
    load_wc(p, sub, w);
    for (; j0 < n_atoms; j0 += step) {
        int64_t nnlo, nnhi;
        row_range(j0 + 2 * step, nnlo, nnhi);
        const int64_t j = j0 + row;
        const bool on = j < n_atoms;
        // component `sub` of the atom's own force and its hosted-WC range, which
        // arrive while the rows are summed
        T own = T(0);
        int h0 = 0, h1 = 0;
        if (on && sub < 3) {
            own = f_sites[3 * j + sub];
            if (host_ptr) {
                h0 = host_ptr[j];
                h1 = host_ptr[j + 1];
            }
        }
        // the next run's first piece
        const int64_t nke = __shfl_sync(0xffffffffu, nhi, 31);
        const Piece np = piece(__shfl_sync(0xffffffffu, nlo, 0), nke, nlo, nhi);
        T a0 = T(0), a1 = T(0), a2 = T(0);
        bool more;
        do {
            const int jl = copy_vectors<CAP * BLOCK>(S.jac, jb + p.k * BLOCK, (int)(p.e - p.k) * BLOCK, jb, je, lane);
            asm volatile("cp.async.commit_group;" ::: "memory");
            const T* J0 = reinterpret_cast<const T*>(S.jac + jl) + 9 * p.b;
            more = p.e < ke;
            const Piece next = more ? piece(p.e, ke, lo, hi) : np;
            for (int i0 = sub;;) {
                T g[U][3];
                bool in[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    in[u] = (unsigned)w[u] < nwc;
                    bad |= !in[u] && i0 + u * G < p.n;
                    g[u][0] = g[u][1] = g[u][2] = T(0);
                    if (in[u]) {
                        const T* f = fw + 3 * (int64_t)w[u];
                        if ((unsigned)w[u] + 1 < nwc) {
                            load_row3(f, g[u][0], g[u][1], g[u][2]);
                        } else {
                            g[u][0] = f[0];
                            g[u][1] = f[1];
                            g[u][2] = f[2];
                        }
                    }
                }
                // the indices of the row's further blocks, or of the next piece
                const int i = i0;
                i0 += U * G;
                const bool last = !__any_sync(0xffffffffu, i0 < p.n);
                load_wc(last ? next : p, last ? sub : i0, w);
                if (i == sub) {
                    asm volatile("cp.async.wait_group 0;" ::: "memory");
                    __syncwarp();
                }
                T c[U][3];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const T* J = J0 + 9 * (i + u * G);
                    // (J^T g)_b = sum_a J[a][b] g_a
#pragma unroll
                    for (int d = 0; d < 3; ++d)
                        c[u][d] = in[u] ? J[d] * g[u][0] + J[3 + d] * g[u][1] + J[6 + d] * g[u][2] : T(0);
                }
#pragma unroll
                for (int h = U / 2; h >= 1; h >>= 1)
#pragma unroll
                    for (int u = 0; u < h; ++u)
#pragma unroll
                        for (int d = 0; d < 3; ++d) c[u][d] += c[u + h][d];
                a0 += c[0][0];
                a1 += c[0][1];
                a2 += c[0][2];
                if (last) break;
            }
            __syncwarp();  // the stage may be filled again
            p = next;
        } while (more);
        for (int h = G >> 1; h >= 1; h >>= 1) {
            a0 += __shfl_xor_sync(0xffffffffu, a0, h);
            a1 += __shfl_xor_sync(0xffffffffu, a1, h);
            a2 += __shfl_xor_sync(0xffffffffu, a2, h);
        }
        if (on) {
            for (int c = sub; c < 3; c += G) {
                T v = c == sub ? own : f_sites[3 * j + c];
                for (int h = h0; h < h1; ++h) {
                    const int w = host_wc[h];
                    if ((unsigned)w < nwc) v += fw[3 * (int64_t)w + c];
                    else bad = true;
                }
                f_atoms[3 * j + c] = v + (c == 0 ? a0 : c == 1 ? a1 : a2);
            }
        }
        lo = nlo;
        hi = nhi;
        ke = nke;
        nlo = nnlo;
        nhi = nnhi;
    }
    if (bad && status) atomicOr(status, 1);
}

template <typename T>
int wc_fold(void* stream, int64_t n_atoms, int64_t n_wc, const T* f_sites, const int* host_ptr, const int* host_wc,
            const int64_t* jac_ptr, const int* jac_wc, const T* jac, T* f_atoms, int* status) {
    if (n_atoms < 0 || n_wc < 0 || (n_atoms > 0 && (!f_sites || !f_atoms))) return PPPM_ERR_INVALID_ARG;
    if ((host_ptr && !host_wc) || (jac_ptr && (!jac_wc || !jac))) return PPPM_ERR_INVALID_ARG;
    if (n_atoms == 0) return PPPM_OK;
    void (*kern)(int64_t, int64_t, const T*, const int*, const int*, const int64_t*, const int*, const T*, T*, int*);
    size_t smem = 0;
    int per = kLaneBlocks;
    if constexpr (sizeof(T) == 4) {
        kern = k_wc_fold_lanes;
    } else {
        kern = k_wc_fold_rows;
        smem = kFoldWarps * sizeof(FoldStage);
        per = kRowBlocks;
    }
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        allow_smem(kern, smem) != cudaSuccess)
        return PPPM_ERR_CUDA;
    int64_t blocks = (n_atoms + kFoldWarps - 1) / kFoldWarps;
    const int64_t cap = (int64_t)nsm * per;  // the resident blocks
    if (blocks > cap) blocks = cap;
    kern<<<(unsigned)blocks, kFoldWarps * 32, smem, (cudaStream_t)stream>>>(n_atoms, n_wc, f_sites, host_ptr, host_wc,
                                                                            jac_ptr, jac_wc, jac, f_atoms, status);
    return cudaGetLastError() == cudaSuccess ? PPPM_OK : PPPM_ERR_CUDA;
}

}  // namespace pppm

extern "C" {

int pppm_wc_fold(void* stream, int64_t n_atoms, int64_t n_wc, const double* f_sites, const int* host_ptr,
                 const int* host_wc, const int64_t* jac_ptr, const int* jac_wc, const double* jac, double* f_atoms,
                 int* status) {
    return pppm::wc_fold<double>(stream, n_atoms, n_wc, f_sites, host_ptr, host_wc, jac_ptr, jac_wc, jac, f_atoms,
                                 status);
}

int pppm_wc_fold_f32(void* stream, int64_t n_atoms, int64_t n_wc, const float* f_sites, const int* host_ptr,
                     const int* host_wc, const int64_t* jac_ptr, const int* jac_wc, const float* jac,
                     float* f_atoms, int* status) {
    return pppm::wc_fold<float>(stream, n_atoms, n_wc, f_sites, host_ptr, host_wc, jac_ptr, jac_wc, jac, f_atoms,
                                status);
}

}  // extern "C"
