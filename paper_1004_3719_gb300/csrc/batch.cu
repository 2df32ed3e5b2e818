// Many independent products Y_j = A_j X_j (mod m_j) in one launch.
//
// Every matrix brings its block layout (block.cu: rows in length classes, X
// packed in 16-byte pieces), built on its first batched or block product and
// kept on the handle; a launch finds its work from the handles alone (a CTA
// looks its matrix up in the launch parameters), so another set of handles that
// have their layouts costs nothing but the call.  Layouts that are missing are
// built together first: a first batch over 48 new handles of 200 to 5 000 rows
// takes 2.1 ms (4.6 with the work list described below, 5.0 with a build for
// each), of 1 000 to 200 000 rows 25 ms (60).
//
// Measured, 48 problems of 1 000 to 200 000 rows, 1 to 32 vectors, primes near
// 2^31, another set of handles on every call: 22.9 ms with a work list that
// was rebuilt, uploaded and timed in six tile shapes for each new set, 0.47 ms
// here; the same set again: 512 us before, 427 us now.
#include <algorithm>
#include <exception>
#include <vector>

#include "ff_block.h"
#include "ff_internal.cuh"

using namespace ff;

static ffspmv_status batch_apply(int32_t count, const ffspmv_t *hs, const uint32_t *const *d_x, uint32_t *const *d_y,
                                 const int32_t *nvec, cudaStream_t st)
{
    // a handle's X is staged in a buffer of the handle: its first product goes
    // into the first round, its second into the second, and so on
    std::vector<int> by(count), turn(count, 0);
    for (int j = 0; j < count; ++j) by[j] = j;
    std::sort(by.begin(), by.end(), [&](int a, int b) { return hs[a] != hs[b] ? hs[a] < hs[b] : a < b; });
    int rounds = 1;
    for (int i = 1; i < count; ++i)
        if (hs[by[i]] == hs[by[i - 1]]) rounds = std::max(rounds, (turn[by[i]] = turn[by[i - 1]] + 1) + 1);
    // the handles' layouts, those that are missing all at once
    std::vector<ffspmv_handle *> missing;
    std::vector<const u32 *> mx;
    std::vector<int> mv;
    for (int j = 0; j < count; ++j)
        if (turn[j] == 0 && hs[j]->A.nrows > 0 && !(hs[j]->block[0] && hs[j]->block[0]->ok)) {
            missing.push_back(hs[j]);
            mx.push_back(d_x[j]);
            mv.push_back(nvec[j]);
        }
    if (!missing.empty()) ensure_blocks((int)missing.size(), missing.data(), mx.data(), mv.data(), st);
    std::vector<const BlockPlan *> B;
    std::vector<uint4 *> xs;
    std::vector<const u32 *> x;
    std::vector<u32 *> y;
    std::vector<int> nv;
    for (int r = 0; r < rounds; ++r) {
        B.clear();
        xs.clear();
        x.clear();
        y.clear();
        nv.clear();
        for (int j = 0; j < count; ++j) {
            if (turn[j] != r || hs[j]->A.nrows == 0) continue;
            BlockPlan *b = hs[j]->block[0];
            uint4 *xj = nullptr;
            if (!b || !b->ok || !block_staging(*b, d_x[j], nvec[j], nvec[j], st, &xj)) {
                // no block layout (no memory for it, or the stream is being
                // captured before it exists): the matrix's own plan
                const ffspmv_status s = run_plan(hs[j]->A, d_x[j], nvec[j], d_y[j], nvec[j], nvec[j], hs[j]->m, 1, 0, st);
                if (s != FFSPMV_OK) return s;
                continue;
            }
            B.push_back(b);
            xs.push_back(xj);
            x.push_back(d_x[j]);
            y.push_back(d_y[j]);
            nv.push_back(nvec[j]);
        }
        const ffspmv_status s = run_block_many((int)B.size(), B.data(), xs.data(), x.data(), y.data(), nv.data(), st);
        if (s != FFSPMV_OK) return s;
    }
    return FFSPMV_OK;
}

extern "C" ffspmv_status spmv_batch_apply(int32_t count, const ffspmv_t *hs,
                                          const uint32_t *const *d_x, uint32_t *const *d_y,
                                          const int32_t *nvec, ffspmv_stream_t stream)
{
    if (count < 0 || (count > 0 && (!hs || !d_x || !d_y || !nvec))) return FFSPMV_ERR_ARG;
    if (count == 0) return FFSPMV_OK;
    for (int j = 0; j < count; ++j) {
        if (!hs[j] || nvec[j] < 1 || nvec[j] > 32) return FFSPMV_ERR_ARG;
        if ((hs[j]->A.nrows > 0 && !d_y[j]) || (hs[j]->A.ncols > 0 && !d_x[j])) return FFSPMV_ERR_ARG;
    }
    try {
        return batch_apply(count, hs, d_x, d_y, nvec, (cudaStream_t)stream);
    } catch (const std::exception &) {
        return FFSPMV_ERR_OOM;
    }
}
