// Shared by the translation units of the batched form: the stages, the
// description of one box and the device buffers of a batch.
#pragma once

#include "internal.cuh"

namespace pppm {
namespace batch {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
enum Stage { S_BIN, S_SCAN, S_SCATTER, S_SPREAD, S_ZR2C, S_YFWD, S_XINF, S_YINV, S_ZC2R, S_GATHER, NSTAGE };
// the FFT stages are S_ZR2C .. S_ZC2R
constexpr int NFFT = S_ZC2R - S_ZR2C + 1;
constexpr int kSiteChunk = 1024;  // sites per bin / scatter item
constexpr int kZPairs = 8;        // row pairs per z-pass item, at least
constexpr int kZRows = 512;       // and up to about this many points (pairs x Nz) an item
constexpr int kSpreadTiles = 2;  // tiles per spread item, one after another by the whole block
constexpr int kGatherTiles = 2;   // four warps per tile

struct BoxDesc {
    Geo g;
    Radix rad[3];
    Bundle bd;
    FieldLayout fl;
    long long site0;
    int nsite;
    int tile0;   // into tile_count
    int ts0;     // into tile_start (ntiles + 1 entries per box)
    long long patch0;
    long long c0;  // complex half-spectrum offset
    long long f0;  // padded field offset (3 fields)
    long long G0;
    int tw0[3];
    int cov0;
    int nmax;
    int part0;
    float e_scale, c_field, beta;
    int zp;  // row pairs per z-pass item
    int nitems[NSTAGE];
    // the staged launch's FFT stages on the register engines (batched_fft.cu)
    int rnitems[NFFT];
    int cov_x0, cov_yz0;  // fold tables (PatchSrc): offsets of this box's entries
    int cov_deep;
    long long xstride;
};

struct Bufs {
    const float* pos;
    const float* q;
    float* forces;
    double* energy;
    double* virial;
    int* tile_count;
    int* tile_start;
    int* tile_of;
    int* slot_of;
    Rec<float>* rec;
    int* cell;
    int* scell;
    int* sorig;
    Rec<float>* srec;  // tile order: the sites' records (B-spline arguments, charge)
    float* patch;
    float2* cx0;
    float2* cx1;
    float2* cx2;
    float* fields;
    const float* G;
    const float2* tw;
    const int4* cov2;
    const int2* cov_x;   // fold tables of the register engines' z pass
    const int4* cov_yz;
    float* partial;
    unsigned int* box_counter;
    int* box_fail;  // set when a wait of the box ran out: its later stages skip their work
    int* status;
    double prefactor;
    int dft_max;  // lines up to this length take the tensor-core DFT (0: all take the FFT)
    int qgroup;     // node size of the int32-quantised DFT (0: off)
    double qscale;  // its scale
    int wait_probe;  // 1: box 0's scan waits for one binning item more than exist (its wait runs out)
    RedRows red_rows;  // lane -> stencil row of the spread's shared-memory atomics
};

// batched_fft.cu: the FFT stages of the staged launch on the register engines
bool reg_fft_length(int L);                                // a line length they serve
int reg_fft_items(int stage, const int N[3], int Hz);      // work items of one box
cudaError_t launch_reg_fft(cudaStream_t s, int stage, const BoxDesc* boxes, const int2* items, int count,
                           const Bufs& B, size_t smem);
size_t reg_fft_smem(int stage, const int N[3]);            // dynamic shared memory one box's items need

}  // namespace batch
}  // namespace pppm
