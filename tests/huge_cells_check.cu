// The kernel of alignment cells whose scores may reach 2^28 (csrc/longpair.cu) on pairs of ordinary
// size, which the library never sends there: passes fewer and more than a CTA's warps, more jobs
// than CTAs, both directions, against the recurrences in three plain rows.  Then a wait that runs
// out: the error is 2 and the next launch is right again.
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>

#include "longpair.cu"

using namespace cm;

#define TRY(call)                                                                          \
    do {                                                                                   \
        const cudaError_t e = (call);                                                      \
        if (e != cudaSuccess) { std::printf("%s: %s\n", #call, cudaGetErrorString(e)); return 2; } \
    } while (0)

static std::vector<int32_t> first_cell(const uint8_t* x, int32_t m, const uint8_t* y, int32_t n, bool rev,
                                       const int16_t* mat, int32_t o, int32_t e)
{
    std::vector<int32_t> H((size_t)n + 1, 0), F((size_t)n + 1, -(1 << 28));
    int32_t best = 0, row = -1, col = -1;
    for (int32_t i = 0; i < m; ++i) {
        int32_t diag = 0, left = 0, E = -(1 << 28);
        for (int32_t j = 0; j < n; ++j) {
            const int s = mat[(rev ? x[m - 1 - i] : x[i]) * kAlpha + (rev ? y[n - 1 - j] : y[j])];
            E = std::max(E - e, left - o);
            F[j + 1] = std::max(F[j + 1] - e, H[j + 1] - o);
            const int32_t h = std::max(std::max(0, diag + s), std::max(E, F[j + 1]));
            diag = H[j + 1];
            H[j + 1] = left = h;
            if (h > best) { best = h; row = i; col = j; }
        }
    }
    return {best, row, col};
}

int main()
{
    std::mt19937 rng(28);
    const std::vector<int32_t> lens = {1, 40, 255, 256, 257, 900, 2049, 2600};
    std::vector<uint8_t> root(2600), db;
    for (auto& v : root) v = (uint8_t)(rng() % 24);
    std::vector<int64_t> off(1, 0);
    for (int32_t n : lens) {
        for (int32_t i = 0; i < n; ++i) db.push_back(rng() % 3 ? root[i] : (uint8_t)(rng() % 24));
        off.push_back((int64_t)db.size());
    }
    SwArgs a{};
    for (int i = 0; i < kAlpha * kAlpha; ++i) a.mat[i] = (int16_t)((int)(rng() % 12) - 8);
    for (int i = 0; i < kAlpha; ++i) a.mat[i * (kAlpha + 1)] = 6;
    a.gap_open = 11;
    a.gap_extend = 1;
    std::vector<CellJob> jobs;
    for (int32_t x = 0; x < (int32_t)lens.size(); ++x)
        for (int32_t y = 0; y < (int32_t)lens.size(); ++y)
            for (int32_t rev = 0; rev < 2; ++rev) jobs.push_back({x, y, lens[x], lens[y], rev, 0});
    const int32_t nj = (int32_t)jobs.size();
    const int grid = 3;
    a.bnd_stride = 2600 + 64;
    uint8_t* d_db;
    int64_t* d_off;
    uint2* d_bnd;
    int32_t *d_words, *d_res;
    CellJob* d_jobs;
    TRY(cudaMalloc(&d_db, db.size()));
    TRY(cudaMalloc(&d_off, off.size() * sizeof(int64_t)));
    TRY(cudaMalloc(&d_bnd, sizeof(uint2) * grid * kLongSlots * a.bnd_stride));
    TRY(cudaMalloc(&d_words, 2 * sizeof(int32_t)));
    TRY(cudaMalloc(&d_res, 3 * sizeof(int32_t) * nj));
    TRY(cudaMalloc(&d_jobs, sizeof(CellJob) * nj));
    TRY(cudaMemcpy(d_db, db.data(), db.size(), cudaMemcpyHostToDevice));
    TRY(cudaMemcpy(d_off, off.data(), off.size() * sizeof(int64_t), cudaMemcpyHostToDevice));
    TRY(cudaMemcpy(d_jobs, jobs.data(), sizeof(CellJob) * nj, cudaMemcpyHostToDevice));
    a.db = d_db;
    a.off = d_off;
    a.bnd = d_bnd;
    a.err = d_words;
    for (int run = 0; run < 3; ++run) {
        a.wait_limit = run == 1 ? 1 : 1 << 24;
        TRY(cudaMemset(d_words, 0, 2 * sizeof(int32_t)));
        TRY(launch_huge_cells(grid, a, d_jobs, nj, d_words + 1, d_res, 0));
        TRY(cudaDeviceSynchronize());
        int32_t err = -1;
        std::vector<int32_t> res((size_t)nj * 3);
        TRY(cudaMemcpy(&err, d_words, sizeof(err), cudaMemcpyDeviceToHost));
        TRY(cudaMemcpy(res.data(), d_res, res.size() * sizeof(int32_t), cudaMemcpyDeviceToHost));
        if (err != (run == 1 ? 2 : 0)) { std::printf("run %d: error %d\n", run, err); return 1; }
        for (int32_t q = 0; run != 1 && q < nj; ++q) {
            const CellJob& J = jobs[q];
            const std::vector<int32_t> want = first_cell(db.data() + off[J.a], J.m, db.data() + off[J.b],
                                                         J.n, J.reverse != 0, a.mat, 11, 1);
            if (std::memcmp(want.data(), &res[3 * (size_t)q], 12) != 0) {
                std::printf("run %d: %d x %d, reverse %d: %d %d %d, not %d %d %d\n", run, J.m, J.n, J.reverse,
                            res[3 * q], res[3 * q + 1], res[3 * q + 2], want[0], want[1], want[2]);
                return 1;
            }
        }
    }
    std::printf("ok\n");
    return 0;
}
