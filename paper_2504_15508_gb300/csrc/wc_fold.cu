// Fold of the Wannier-centroid forces onto atoms, Eq. DPLR:F_final.
//
// W_n = R_host(n) + Delta_n(R) (Eq. DPLR:Wn), so the long-range force on atom j
// is its own site force, plus the force on every WC it hosts, plus
// J^T F_W(n) for every Jacobian block J = dDelta_n/dR_j listed in its row.
// A warp takes runs of kFoldRun consecutive atoms, whose rows are one
// contiguous run of blocks.  It streams them in chunks of 32 blocks, one a
// lane, through a small ring in shared memory (cp.async, kStages - 1 chunks
// ahead): read in place, a lane's nine values lie 36 bytes from its
// neighbour's, so that each of the nine loads touches nine cache lines, while
// the ring is filled by whole 16-byte vectors and read with an odd stride free
// of bank conflicts.  The WC force of the next chunk's blocks, the one
// scattered read, is fetched while the current chunk is summed.  Each block is
// added to its row's accumulator in its lane, and four rows at a time are
// summed over the lanes by a transposing butterfly (16 shuffles), which leaves
// component c of row r in lane 4 r + c; that lane adds the atom's own force
// and those of the WCs it hosts, in row order.  Every sum has a fixed order:
// the result is bitwise reproducible.
//
// Bound by the scattered reads of the WC forces (12 bytes each from L2, a cache
// line a lane) and the instructions of the sums; the stream of 40 B a block in
// FP32 alone would take 34 us at 6.8 TB/s.  72,192 molecules (216,576 atoms,
// up to 27 blocks each), FP32: 90.6 us with the blocks read in place and the
// butterfly over eight lanes an atom; 89.0 with the ring alone, 77.9 with whole
// runs and the transposing sum; eight lanes a row on a double-buffered ring
// took 91.0.
#include <cstdint>

#include "internal.cuh"

namespace pppm {

constexpr int kFoldWarps = 8;
constexpr int kFoldRun = 16;  // atoms a warp takes at a time
constexpr int kStages = 4;    // chunks in the ring

template <typename T>
struct FoldStage {
    // 32 blocks and the bytes before the first one in its 16-byte vector
    __align__(16) unsigned char jac[32 * 9 * sizeof(T) + 16];
    int wc[32];
};

template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst, const void* src) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(BYTES) : "memory");
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

template <typename T>
__global__ void __launch_bounds__(kFoldWarps * 32, sizeof(T) == 4 ? 4 : 3)
k_wc_fold(int64_t n_atoms, int64_t n_wc, const T* __restrict__ f_sites, const int* __restrict__ host_ptr,
          const int* __restrict__ host_wc, const int64_t* __restrict__ jac_ptr, const int* __restrict__ jac_wc,
          const T* __restrict__ jac, T* __restrict__ f_atoms, int* __restrict__ status) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    typedef FoldStage<T> Stage;
    constexpr int BLOCK = 9 * (int)sizeof(T), CHUNK = 32 * BLOCK, WHOLE = CHUNK / 16;  // bytes; vectors of a chunk
    Stage* ring = reinterpret_cast<Stage*>(smem_raw) + (threadIdx.x >> 5) * kStages;
    const int lane = threadIdx.x & 31;
    const int64_t runs = (n_atoms + kFoldRun - 1) / kFoldRun;
    const int64_t warps = (int64_t)gridDim.x * kFoldWarps;
    const T* fw = f_sites + 3 * n_atoms;
    // whole 16-byte vectors where the Jacobian starts on one, else value by value
    const bool vec = (reinterpret_cast<uintptr_t>(jac) & 15) == 0;
    bool bad = false;
    for (int64_t run = (int64_t)blockIdx.x * kFoldWarps + (threadIdx.x >> 5); run < runs; run += warps) {
        const int64_t j0 = run * kFoldRun;
        const int na = (int)min((int64_t)kFoldRun, n_atoms - j0);
        // lane i: where row i of the run starts (the run's end from i = na on)
        const int64_t ptr = jac_ptr ? jac_ptr[j0 + min(lane, na)] : 0;
        const int64_t kb = __shfl_sync(0xffffffffu, ptr, 0), ke = __shfl_sync(0xffffffffu, ptr, 31);
        // this lane's next vector of the Jacobian, and the next index; chunks are
        // whole vectors, so the bytes before a chunk in its first one are the same
        // for every chunk of the run
        const char* src = reinterpret_cast<const char*>(jac + 9 * kb);
        const int lead = vec ? (int)(reinterpret_cast<uintptr_t>(src) & 15) : 0;
        const char* src16 = src - lead + 16 * lane;
        const int* srcw = jac_wc + kb + lane;
        int64_t left = ke - kb;  // blocks not yet asked for
        int in = 0;              // stage of the next fill
        auto fill = [&]() {      // the next chunk into the ring (one cp.async group)
            Stage& st = ring[in];
            if (left >= 32 && vec) {
                cp_async<16>(st.jac + 16 * lane, src16);
                cp_async<16>(st.jac + 16 * (lane + 32), src16 + 512);
#pragma unroll
                for (int v = 64; v < WHOLE; v += 32)
                    if (v + 32 <= WHOLE || lane < WHOLE - v) cp_async<16>(st.jac + 16 * (lane + v), src16 + 16 * v);
                // the last block's values past the last whole vector
                if (lane * (int)sizeof(T) < lead)
                    cp_async<sizeof(T)>(st.jac + CHUNK + lane * sizeof(T), src16 + CHUNK - 16 * lane + lane * sizeof(T));
                cp_async<4>(&st.wc[lane], srcw);
            } else if (left > 0) {
                const int nb = (int)min((int64_t)32, left);
                const char* s0 = src16 - 16 * lane + lead;
                for (int v = lane; v < 9 * nb; v += 32)
                    cp_async<sizeof(T)>(st.jac + lead + v * sizeof(T), s0 + v * sizeof(T));
                if (lane < nb) cp_async<4>(&st.wc[lane], srcw);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
            src16 += CHUNK;
            srcw += 32;
            left -= 32;
            in = in + 1 == kStages ? 0 : in + 1;
        };
        __syncwarp();  // the previous run's chunks have been read
#pragma unroll
        for (int c = 0; c < kStages - 1; ++c) fill();
        int out = 0;                        // stage of the next chunk
        int64_t k0 = kb;                    // the next chunk's first block
        int64_t kc = kb - 32;               // the current chunk's first block
        T c0 = T(0), c1 = T(0), c2 = T(0);  // the terms of its block `lane`
        T g0 = T(0), g1 = T(0), g2 = T(0);  // WC force of the next chunk's block
        auto fetch = [&]() {
            g0 = g1 = g2 = T(0);
            if (k0 + lane < ke) {
                const int n = ring[out].wc[lane];
                if (n < 0 || n >= n_wc) {
                    bad = true;
                } else if (n + 1 < n_wc) {
                    load_row3(fw + 3 * (int64_t)n, g0, g1, g2);
                } else {
                    g0 = fw[3 * (int64_t)n];
                    g1 = fw[3 * (int64_t)n + 1];
                    g2 = fw[3 * (int64_t)n + 2];
                }
            }
        };
        asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
        __syncwarp();
        fetch();
        auto advance = [&]() {  // the next chunk becomes the current one
            const T h0 = g0, h1 = g1, h2 = g2;
            const T* J = reinterpret_cast<const T*>(ring[out].jac + lead) + 9 * lane;
            const bool any = k0 + lane < ke;
            kc = k0;
            k0 += 32;
            out = out + 1 == kStages ? 0 : out + 1;
            fill();  // into the stage of the chunk before this one
            asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");  // the next chunk has landed
            __syncwarp();
            fetch();
            // (J^T g)_b = sum_a J[a][b] g_a
            c0 = any ? J[0] * h0 + J[3] * h1 + J[6] * h2 : T(0);
            c1 = any ? J[1] * h0 + J[4] * h1 + J[7] * h2 : T(0);
            c2 = any ? J[2] * h0 + J[5] * h1 + J[8] * h2 : T(0);
            __syncwarp();  // this stage is refilled by the next advance
        };
        int64_t lo = kb;  // the next block to be summed
        for (int q = 0; q < na; q += 4) {
            // lane 4 r + c: component c of atom j0 + q + r, its own force and
            // hosted-WC range, loaded before the rows so that they arrive meanwhile
            const int r4 = q + ((lane & 15) >> 2), comp = lane & 3;
            const int64_t j = j0 + r4;
            const bool mine = lane < 16 && comp < 3 && r4 < na;
            T own = T(0);
            int h0 = 0, h1 = 0;
            if (mine) {
                own = f_sites[3 * j + comp];
                if (host_ptr) {
                    h0 = host_ptr[j];
                    h1 = host_ptr[j + 1];
                }
            }
            T acc[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) acc[i] = T(0);
            if (kb < ke) {
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int64_t hi = __shfl_sync(0xffffffffu, ptr, min(q + r + 1, 31));
                    while (lo < hi) {
                        if (lo >= kc + 32) advance();
                        const int first = (int)(lo - kc), last = (int)min(hi - kc, (int64_t)32);
                        if (lane >= first && lane < last) {
                            acc[4 * r] += c0;
                            acc[4 * r + 1] += c1;
                            acc[4 * r + 2] += c2;
                        }
                        lo = kc + last;
                    }
                }
#pragma unroll
                for (int h = 8; h >= 1; h >>= 1) {
                    const bool up = (lane & h) != 0;
#pragma unroll
                    for (int i = 0; i < h; ++i) {
                        const T send = up ? acc[i] : acc[i + h];
                        const T keep = up ? acc[i + h] : acc[i];
                        acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, h);
                    }
                }
                acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 16);
            }
            if (mine) {
                for (int h = h0; h < h1; ++h) {
                    const int n = host_wc[h];
                    if (n < 0 || n >= n_wc) bad = true;
                    else own += fw[3 * (int64_t)n + comp];
                }
                f_atoms[3 * j + comp] = own + acc[0];
            }
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    if (bad && status) atomicOr(status, 1);
}

template <typename T>
int wc_fold(void* stream, int64_t n_atoms, int64_t n_wc, const T* f_sites, const int* host_ptr, const int* host_wc,
            const int64_t* jac_ptr, const int* jac_wc, const T* jac, T* f_atoms, int* status) {
    if (n_atoms < 0 || n_wc < 0 || (n_atoms > 0 && (!f_sites || !f_atoms))) return PPPM_ERR_INVALID_ARG;
    if ((host_ptr && !host_wc) || (jac_ptr && (!jac_wc || !jac))) return PPPM_ERR_INVALID_ARG;
    if (n_atoms == 0) return PPPM_OK;
    int dev = 0, nsm = 0, per = 0;
    constexpr size_t smem = kFoldWarps * kStages * sizeof(FoldStage<T>);
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaFuncSetAttribute(k_wc_fold<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_wc_fold<T>, kFoldWarps * 32, smem) != cudaSuccess ||
        per < 1)
        return PPPM_ERR_CUDA;
    int64_t blocks = ((n_atoms + kFoldRun - 1) / kFoldRun + kFoldWarps - 1) / kFoldWarps;
    const int64_t cap = (int64_t)nsm * per;  // the resident blocks
    if (blocks > cap) blocks = cap;
    k_wc_fold<T><<<(unsigned)blocks, kFoldWarps * 32, smem, (cudaStream_t)stream>>>(
        n_atoms, n_wc, f_sites, host_ptr, host_wc, jac_ptr, jac_wc, jac, f_atoms, status);
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
