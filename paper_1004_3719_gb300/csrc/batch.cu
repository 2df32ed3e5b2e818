// Many independent products Y_j = A_j X_j (mod m_j) in one launch.
//
// Every matrix brings its block layout (block.cu: rows in length classes, X
// packed in 16-byte pieces), built on its first batched or block product and
// kept on the handle; a launch finds its work from the handles alone (a CTA
// looks its matrix up in the launch parameters), so another set of handles that
// have their layouts costs nothing but the call.  Layouts that are missing are
// built together first: a first batch over 48 new handles of 200 to 5 000 rows
// takes 1.9 ms (4.6 with the work list described below, 5.0 with a build for
// each), of 1 000 to 200 000 rows 13 ms (60).
//
// Measured, 48 problems of 1 000 to 200 000 rows, 1 to 32 vectors, primes near
// 2^31, handles with their layouts, another set on every call: 23.4 ms with a work
// list that was rebuilt, uploaded and timed in six tile shapes for each new set,
// 0.41 ms here; the same set again 0.51 ms and 0.41.
#include <algorithm>
#include <exception>
#include <vector>

#include "ff_block.h"
#include "ff_internal.cuh"

using namespace ff;

static ffspmv_status batch_apply(int32_t count, const ffspmv_t *hs, const uint32_t *const *d_x, uint32_t *const *d_y,
                                 const int32_t *nvec, cudaStream_t st)
{
    std::vector<int> by(count);   // the products, those of one handle together
    for (int j = 0; j < count; ++j) by[j] = j;
    std::sort(by.begin(), by.end(), [&](int a, int b) { return hs[a] != hs[b] ? hs[a] < hs[b] : a < b; });
    auto same = [&](int i) { return i > 0 && hs[by[i]] == hs[by[i - 1]]; };
    // the handles' layouts, those that are missing all at once
    std::vector<ffspmv_handle *> missing;
    std::vector<const u32 *> mx;
    std::vector<int> mv;
    for (int i = 0; i < count; ++i) {
        const int j = by[i];
        if (same(i) || hs[j]->A.nrows == 0 || (hs[j]->block[0] && hs[j]->block[0]->ok)) continue;
        missing.push_back(hs[j]);
        mx.push_back(d_x[j]);
        mv.push_back(nvec[j]);
    }
    if (!missing.empty()) ensure_blocks((int)missing.size(), missing.data(), mx.data(), mv.data(), st);
    // A handle's products share its staging buffer and the words of its long
    // rows; what does not fit beside the others goes into a later round.  64
    // products with a 2 000 x 2 000 matrix, 8 vectors each: 528 us with a round
    // for each (80 with the former work list), 82 so
    std::vector<int> round(count, -1), v0(count, 0);   // -1: no layout (or no staging) now, the matrix's own plan
    std::vector<uint4 *> xs(count, nullptr);
    int rounds = 0;
    for (int i = 0, end; i < count; i = end) {
        for (end = i + 1; end < count && same(end);) ++end;
        BlockPlan *b = hs[by[i]]->block[0];
        if (hs[by[i]]->A.nrows == 0 || !b || !b->ok) continue;
        int most = 0, total = 0, room = 0;
        for (int k = i; k < end; ++k) {
            const int p = block_pieces(*b, d_x[by[k]], nvec[by[k]]);
            most = std::max(most, p);
            total = std::min(total + p, kBlockPieces);
        }
        uint4 *buf = most ? block_staging(*b, most, total, st, &room) : nullptr;
        int r = 0, pieces = 0, vecs = 0;
        for (int k = i; k < end; ++k) {
            const int j = by[k], p = block_pieces(*b, d_x[j], nvec[j]);
            if (p && !buf) continue;
            if (pieces + p > room || (b->nchunk && vecs + nvec[j] > kBlockVecs)) {
                ++r;
                pieces = vecs = 0;
            }
            round[j] = r;
            if (p) xs[j] = buf + b->ncols * pieces;
            if (b->nchunk) v0[j] = vecs;
            pieces += p;
            vecs += nvec[j];
            rounds = std::max(rounds, r + 1);
        }
    }
    for (int j = 0; j < count; ++j) {
        if (round[j] >= 0 || hs[j]->A.nrows == 0) continue;
        PanelCtl ctl;   // an x-panel plan's waits report to the handle, as in spmv_apply
        ctl.status = hs[j]->d_status + 2;
        ctl.skip_stage = (hs[j]->opt.test_hooks & 2) ? 1 : -1;
        const ffspmv_status s = run_plan(hs[j]->A, d_x[j], nvec[j], d_y[j], nvec[j], nvec[j], hs[j]->m, 1, 0, st, &ctl);
        if (s != FFSPMV_OK) return s;
    }
    std::vector<const BlockPlan *> B;
    std::vector<uint4 *> rx;
    std::vector<const u32 *> x;
    std::vector<u32 *> y;
    std::vector<int> nv, rv;
    for (int r = 0; r < rounds; ++r) {
        B.clear();
        rx.clear();
        x.clear();
        y.clear();
        nv.clear();
        rv.clear();
        for (int j = 0; j < count; ++j) {
            if (round[j] != r) continue;
            B.push_back(hs[j]->block[0]);
            rx.push_back(xs[j]);
            x.push_back(d_x[j]);
            y.push_back(d_y[j]);
            nv.push_back(nvec[j]);
            rv.push_back(v0[j]);
        }
        const ffspmv_status s = run_block_many((int)B.size(), B.data(), rx.data(), x.data(), y.data(), nv.data(), rv.data(), st);
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
