// qr_plan.h -- the TSQR trees of TT-rounding: how a matrix's rows are cut into chunks
// and levels, and the buffers of a tree, handed out of the handle's scratch.  Host
// arithmetic only.
#pragma once
#include <algorithm>
#include <cstddef>
#include <vector>

namespace wg {

// A TSQR tree: level 0 factors chunks of the matrix's rows, each further level
// groups of the R factors of the one before, until one R is left.
struct QRPlan {
    struct Level {
        long long m = 0, rows = 0;  // rows of the level's matrix, rows per chunk
        int C = 1, sub = 1;         // chunks, sub-blocks per chunk
        double *A = nullptr, *tau = nullptr, *R = nullptr, *X = nullptr;  // (X: the stack of the chunks' top rows)
    };
    int k = 0, b = 32;
    std::vector<Level> L;
    std::vector<Level> buf;  // the buffers taken for it (C: R factors, sub: sub-blocks they hold)
    double *T = nullptr;
};
constexpr int QR_MAXL = 24;  // levels at most (a matrix of 2^27 rows takes 15)

// Rows of a sub-block.
inline int qr_block(int k) { return k <= 32 ? 32 : (k + 31) / 32 * 32; }

// The levels above a level 0 of q.L[0].C chunks: g R factors per chunk.
inline void qr_merge_levels(QRPlan &q, int g)
{
    while (q.L.back().C > 1) {
        const int C = q.L.back().C;
        QRPlan::Level l;
        l.m = (long long)C * q.k;
        l.C = (C + g - 1) / g;
        l.sub = g;
        l.rows = (long long)g * q.k;
        q.L.push_back(l);
    }
}

// Chunks that a plan for m rows starts from; it takes this many or fewer.  (This bound
// grows with m; the number a plan takes does not: 64 x 100 + 1 rows of 32 columns in
// chunks of 64 end at 97, where the last chunk has 32 rows, 64 x 100 take 100.)
inline int qr_most_chunks(long long m, int k, int spc)
{
    const long long per = (long long)spc * qr_block(k);
    return (int)std::max(1LL, (m + per - 1) / per);
}

// Sub-blocks of b >= k rows, at most spc per chunk, every chunk at least k rows
// long when there are several; then g R factors per chunk: two where the batch is
// small (the tree's depth is the time), four where it fills the GPU.
inline void qr_plan(QRPlan &q, long long m, int k, int spc, int g)
{
    q.k = k;
    q.b = qr_block(k);
    q.L.clear();
    QRPlan::Level l;
    l.m = m;
    for (int C = qr_most_chunks(m, k, spc);; --C) {
        const long long cr = (m + C - 1) / C;
        if (C == 1 || (cr >= k && m - (long long)(C - 1) * cr >= k)) {
            l.C = C;
            l.rows = std::max(1LL, cr);
            break;
        }
    }
    l.sub = (int)((l.rows + q.b - 1) / q.b);
    q.L.push_back(l);
    qr_merge_levels(q, g);
}

struct Bump {  // counts (base == nullptr) or hands out 256-byte aligned pieces
    char *base = nullptr;
    size_t off = 0;
    template <class T> T *take(size_t n)
    {
        off = (off + 255) & ~size_t(255);
        T *p = base ? reinterpret_cast<T *>(base + off) : nullptr;
        off += sizeof(T) * n;
        return p;
    }
};

// Buffers for the QR of an m x k matrix and for applying it to p columns, also for
// any smaller m of the same k, spc and g: level 0 for the most chunks that any of them
// takes, the levels above for as many R factors as those leave.
inline void qr_take(Bump &bp, QRPlan &q, long long m, int k, int spc, int g, int p)
{
    QRPlan big;
    big.k = k;
    big.L.resize(1);
    big.L[0].C = qr_most_chunks(m, k, spc);
    qr_merge_levels(big, g);
    q.buf.assign(big.L.size(), QRPlan::Level());
    for (size_t l = 0; l < big.L.size(); ++l) {
        QRPlan::Level &v = q.buf[l];
        v.C = big.L[l].C;
        // level 0: C chunks of ceil(m / C) rows, each cut into sub-blocks of its own
        v.sub = l == 0 ? (int)(m / qr_block(k)) + 2 * v.C : v.C * g;
        v.tau = bp.take<double>((size_t)v.sub * k);
        v.R = bp.take<double>((size_t)v.C * k * k);
        if (l > 0) v.X = bp.take<double>((size_t)big.L[l - 1].C * k * p);
    }
}

// Points a plan at its buffers (A: the matrix); false if they do not hold it.
inline bool qr_bind(QRPlan &q, double *A)
{
    if (q.L.size() > q.buf.size()) return false;
    for (size_t l = 0; l < q.L.size(); ++l) {
        if (q.L[l].C > q.buf[l].C || (long long)q.L[l].C * q.L[l].sub > q.buf[l].sub) return false;
        q.L[l].A = l == 0 ? A : q.buf[l - 1].R;
        q.L[l].tau = q.buf[l].tau;
        q.L[l].R = q.buf[l].R;
        q.L[l].X = q.buf[l].X;
    }
    q.T = q.L.back().R;
    return true;
}

}  // namespace wg
