// sw_cells_batch_noalloc: an allocation-free variant of sw_cells_batch.
//
// Who needs it: callers that cannot allocate device memory at call time.  Examples are a
// service whose GPU memory was reserved up front by another framework's caching allocator
// (a fresh cudaMalloc would fail or fragment that pool), and a latency-bound loop that must
// not pay the device-wide synchronisation cudaMalloc / cudaFree can cause.  Such callers
// pass device inputs and outputs; the per-pair DP rows live in one fixed array compiled into
// this library instead of a context's grow-on-demand buffers.
//
// The scratch below is a file-scope __device__ array.  In host code its name is only a
// host-side stand-in, never a device address, so every call looks up the real address with
// cudaGetSymbolAddress (with the caller's device current) and passes that pointer to the
// kernels.  The address is not cached: after a cudaDeviceReset the module is loaded again and
// the array may move, and a lookup allocates nothing.  Every GPU that loads the library holds
// the array until the process exits.  All calls on a device share it, so two calls whose work
// overlaps on the GPU race; the array keeps the last call's contents, and the status words at
// its end are cleared at the start of every call.
#include <algorithm>
#include <cstdio>
#include <cstring>

#include "cm_internal.h"
#include "wave32.cuh"

namespace cm {
namespace {

constexpr int kNaWarps = 1024;                   // pairs in flight (one warp each)
constexpr int kNaCols = 4096;                    // boundary row length: second sequence <= 4095
constexpr size_t kNaRowWords = 2ull * kNaWarps * kNaCols;     // H and E rows: 32 MiB
constexpr size_t kNaStatusWords = 64;            // status words after the rows

static __device__ __align__(256) int32_t g_na_scratch[kNaRowWords + kNaStatusWords];

struct NaMatrix {
    int16_t v[400];
};

void na_message(char* buf, int32_t len, const char* msg)
{
    if (buf && len > 0) {
        std::strncpy(buf, msg, (size_t)len - 1);
        buf[len - 1] = '\0';
    }
}

// status[0]: pair index out of range or bad offsets; status[1]: second sequence too long;
// status[2]: residue code >= 20.  One warp per pair.
__global__ void na_check_kernel(const uint8_t* __restrict__ seqs, const int64_t* __restrict__ off,
                                int32_t n_seqs, const int32_t* __restrict__ pairs, int64_t npairs,
                                int32_t* status)
{
    const int lane = threadIdx.x & 31;
    for (int64_t p = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; p < npairs;
         p += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int32_t x = pairs[2 * p], y = pairs[2 * p + 1];
        if (x < 0 || x >= n_seqs || y < 0 || y >= n_seqs) { atomicExch(status + 0, 1); continue; }
        const int64_t xb = off[x], xe = off[x + 1], yb = off[y], ye = off[y + 1];
        if (xb < 0 || xe < xb || yb < 0 || ye < yb) { atomicExch(status + 0, 1); continue; }
        if (ye - yb > kNaCols - 1) { atomicExch(status + 1, 1); continue; }
        bool bad = false;
        for (int64_t i = xb + lane; i < xe; i += 32) bad |= seqs[i] >= 20;
        for (int64_t i = yb + lane; i < ye; i += 32) bad |= seqs[i] >= 20;
        if (bad) atomicExch(status + 2, 1);
    }
}

// Optimum of a[0..m) x b[0..n) (both back to front when `rev`) and its first row-major cell,
// 1-based (0 when the score is 0).  wave32.cuh's wavefront with the rows held (strips of 256,
// eight per lane) and the columns streamed: a strip hands its last row to the next through the
// warp's boundary row, at most 4,095 pairs of words however long the first sequence is.
__device__ int32_t na_optimum(const uint8_t* a, int64_t m, const uint8_t* b, int32_t n, bool rev,
                              const int8_t* mat, int32_t g1, int32_t ge, uint2* prof, int2* bnd,
                              int32_t* bi, int32_t* bj)
{
    constexpr int kRowsHeld = 32 * kWaveMaxR;
    WaveStrip s;
    s.prof = prof;
    s.x = b;
    s.xn = n;
    s.reverse = rev;
    s.o = g1;
    s.ge = ge;
    int32_t best = 0, row = -1, col = -1;
    auto no_wait = [](int32_t) { return true; };
    auto no_publish = [](int32_t) {};
    for (int64_t i0 = 0; i0 < m && n > 0; i0 += kRowsHeld) {
        s.bin = i0 > 0 ? bnd : nullptr;
        s.bout = i0 + kRowsHeld < m ? bnd : nullptr;
        s.y0 = (int32_t)i0;
        __syncwarp();
        wave_profile(prof, a, m, rev, i0, kWaveMaxR, mat, 20, 1, 20);
        __syncwarp();
        int32_t sc, x, y;
        wave_strip<kWaveMaxR, kTrackYRows>(s, no_wait, no_publish, sc, x, y);
        if (first_max(sc, y, x, best, row, col)) { best = sc; row = y; col = x; }
    }
    *bi = row + 1;
    *bj = col + 1;
    return best;
}

// One warp per pair, pairs taken from a queue.  Bound by the serial chain of the longest pairs;
// 200 pairs of up to 600 residues: 0.58 ms per call, 252 ms with one thread per pair and its
// rows in the scratch array.
__global__ void __launch_bounds__(32) na_cells_kernel(const uint8_t* __restrict__ seqs,
                                                      const int64_t* __restrict__ off,
                                                      const int32_t* __restrict__ pairs,
                                                      int64_t npairs, const NaMatrix mat_in,
                                                      int32_t g1, int32_t ge,
                                                      int32_t* __restrict__ cells,
                                                      int32_t* scratch, int32_t* ticket)
{
    __shared__ int8_t mat[400];
    __shared__ uint2 prof[kWaveProf];
    const int lane = threadIdx.x;
    for (int i = lane; i < 400; i += 32) mat[i] = (int8_t)mat_in.v[i];
    __syncwarp();
    int2* bnd = reinterpret_cast<int2*>(scratch) + (size_t)blockIdx.x * kNaCols;
    for (;;) {
        uint32_t p = 0;
        if (lane == 0) p = (uint32_t)atomicAdd(ticket, 1);
        p = __shfl_sync(0xffffffffu, p, 0);
        if (p >= npairs) break;
        const int32_t x = pairs[2 * (int64_t)p], y = pairs[2 * (int64_t)p + 1];
        const uint8_t* a = seqs + off[x];
        const uint8_t* b = seqs + off[y];
        const int64_t m = off[x + 1] - off[x];
        const int32_t n = (int32_t)(off[y + 1] - off[y]);
        int32_t ie, je, ri = 0, rj = 0;
        const int32_t best = na_optimum(a, m, b, n, false, mat, g1, ge, prof, bnd, &ie, &je);
        if (best > 0) na_optimum(a, ie, b, je, true, mat, g1, ge, prof, bnd, &ri, &rj);
        if (lane == 0) {
            int32_t* c = cells + 5 * (int64_t)p;
            c[0] = best;
            c[1] = best > 0 ? ie - ri + 1 : 0;
            c[2] = best > 0 ? ie : 0;
            c[3] = best > 0 ? je - rj + 1 : 0;
            c[4] = best > 0 ? je : 0;
        }
    }
}

}  // namespace
}  // namespace cm

using namespace cm;

extern "C" int sw_cells_batch_noalloc(const uint8_t* seqs, const int64_t* offsets,
                                      int32_t n_seqs, const int32_t* pairs, int64_t n_pairs,
                                      const int8_t* matrix, int32_t gap_open,
                                      int32_t gap_extend, int32_t* cells_out, void* cuda_stream,
                                      uint32_t flags, char* err_msg, int32_t err_len)
{
    na_message(err_msg, err_len, "");
    if (flags & ~(uint32_t)CM_GAP_BLAST) {
        na_message(err_msg, err_len, "only CM_GAP_BLAST is accepted (inputs are device pointers)");
        return CM_ERR_ARG;
    }
    if (n_seqs < 0 || n_pairs < 0 || n_pairs >= ((int64_t)1 << 31) || !offsets || !matrix ||
        (n_pairs > 0 && (!seqs || !pairs || !cells_out))) {
        na_message(err_msg, err_len, "null pointer or size out of range (n_pairs < 2^31)");
        return CM_ERR_ARG;
    }
    const int64_t g1 = (flags & CM_GAP_BLAST) ? (int64_t)gap_open + gap_extend : gap_open;
    if (g1 < 1 || g1 > 1000 || gap_extend < 0 || gap_extend > g1) {
        na_message(err_msg, err_len, "gap costs must satisfy 1 <= first-gap cost <= 1000 and "
                                     "0 <= gap_extend <= first-gap cost");
        return CM_ERR_ARG;
    }
    NaMatrix M;
    for (int i = 0; i < 400; ++i) {
        if (matrix[i] < -1000 || matrix[i] > 1000) {
            na_message(err_msg, err_len, "matrix entries must lie in [-1000, 1000]");
            return CM_ERR_ARG;
        }
        M.v[i] = matrix[i];
    }
    if (n_pairs == 0) return CM_OK;

    // the array's device address on the current device, looked up on every call
    int32_t* scratch = nullptr;
    {
        void* p = nullptr;
        const cudaError_t le = cudaGetSymbolAddress(&p, g_na_scratch);
        if (le != cudaSuccess || !p) {
            cudaGetLastError();
            na_message(err_msg, err_len, "cudaGetSymbolAddress of the scratch array failed "
                                         "(no usable current CUDA device?)");
            return CM_ERR_CUDA;
        }
        scratch = static_cast<int32_t*>(p);
    }
    int32_t* status = scratch + kNaRowWords;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);

    cudaError_t e = cudaMemsetAsync(status, 0, kNaStatusWords * sizeof(int32_t), st);
    if (e == cudaSuccess) {
        const int64_t blocks = std::min<int64_t>((n_pairs + 7) / 8, 4096);
        na_check_kernel<<<(unsigned)blocks, 256, 0, st>>>(seqs, offsets, n_seqs, pairs, n_pairs,
                                                           status);
        e = cudaGetLastError();
    }
    int32_t hs[3] = {0, 0, 0};
    if (e == cudaSuccess) e = cudaMemcpyAsync(hs, status, sizeof(hs), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        na_message(err_msg, err_len, cudaGetErrorString(e));
        return CM_ERR_CUDA;
    }
    if (hs[0]) {
        na_message(err_msg, err_len, "pair index out of range or offsets not non-decreasing");
        return CM_ERR_ARG;
    }
    if (hs[1]) {
        na_message(err_msg, err_len, "a pair's second sequence is longer than 4095 residues, "
                                     "the fixed scratch limit of this entry point");
        return CM_ERR_ARG;
    }
    if (hs[2]) {
        na_message(err_msg, err_len, "residue code >= 20 in a paired sequence");
        return CM_ERR_RESIDUE;
    }
    na_cells_kernel<<<(unsigned)std::min<int64_t>(n_pairs, kNaWarps), 32, 0, st>>>(
        seqs, offsets, pairs, n_pairs, M, (int32_t)g1, gap_extend, cells_out, scratch, status + 8);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        na_message(err_msg, err_len, cudaGetErrorString(e));
        return CM_ERR_CUDA;
    }
    return CM_OK;
}
