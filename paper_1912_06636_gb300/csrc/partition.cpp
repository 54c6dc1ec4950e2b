// Host-side set-up steps of nao_grid_create: the batch partition and the radial splines.
#include <algorithm>
#include <cmath>

#include "nao_internal.h"

namespace {

struct Keyed {
    double key;
    int64_t idx;
};

inline bool keyed_less(const Keyed &a, const Keyed &b) { return a.key < b.key || (a.key == b.key && a.idx < b.idx); }

struct Splitter {
    const double *xyz;
    int64_t B;
    std::vector<Keyed> tmp;
    std::vector<int64_t> *perm;
    std::vector<int64_t> *offsets;

    // Batches leave in depth-first order. A leaf keeps the order its parent's cut gave it:
    // ascending (coordinate along the parent's axis, index); the root leaf keeps input order.
    void run(int64_t *S, int64_t n, int parent_axis) {
        const int64_t k = (n + B - 1) / B;
        if (k <= 1) {
            if (parent_axis >= 0) {
                for (int64_t i = 0; i < n; i++) tmp[i] = {xyz[3 * S[i] + parent_axis], S[i]};
                std::sort(tmp.begin(), tmp.begin() + n, keyed_less);
                for (int64_t i = 0; i < n; i++) S[i] = tmp[i].idx;
            }
            perm->insert(perm->end(), S, S + n);
            offsets->push_back((int64_t)perm->size());
            return;
        }
        double lo[3], hi[3];
        for (int c = 0; c < 3; c++) lo[c] = hi[c] = xyz[3 * S[0] + c];
        for (int64_t i = 1; i < n; i++)
            for (int c = 0; c < 3; c++) {
                const double v = xyz[3 * S[i] + c];
                lo[c] = v < lo[c] ? v : lo[c];
                hi[c] = v > hi[c] ? v : hi[c];
            }
        int ax = 0;
        for (int c = 1; c < 3; c++)
            if (hi[c] - lo[c] > hi[ax] - lo[ax]) ax = c;
        const int64_t nL = (n * (k / 2)) / k;
        for (int64_t i = 0; i < n; i++) tmp[i] = {xyz[3 * S[i] + ax], S[i]};
        // only the set that goes left matters here: the n_L smallest keys
        std::nth_element(tmp.begin(), tmp.begin() + nL, tmp.begin() + n, keyed_less);
        for (int64_t i = 0; i < n; i++) S[i] = tmp[i].idx;
        run(S, nL, ax);
        run(S + nL, n - nL, ax);
    }
};

}  // namespace

int64_t nao_partition(int64_t n, const double *xyz, int64_t B, std::vector<int64_t> &offsets,
                      std::vector<int64_t> &perm) {
    offsets.assign(1, 0);
    perm.clear();
    perm.reserve((size_t)n);
    std::vector<int64_t> S((size_t)n);
    for (int64_t i = 0; i < n; i++) S[(size_t)i] = i;
    Splitter sp{xyz, B, std::vector<Keyed>((size_t)n), &perm, &offsets};
    sp.run(S.data(), n, -1);
    return (int64_t)offsets.size() - 1;
}

// Natural cubic spline through (k, y_k): second derivatives from the tridiagonal system
// M_{k-1} + 4 M_k + M_{k+1} = 6 (y_{k+1} - 2 y_k + y_{k-1}), M_0 = M_{n-1} = 0 (forward
// elimination, back substitution), then per segment the polynomial in t = s - k:
// y_k + c1 t + c2 t^2 + c3 t^3 with c1 = dy - (2 M_k + M_{k+1})/6, c2 = M_k/2,
// c3 = (M_{k+1} - M_k)/6.
void nao_spline_coefficients(const double *y, int32_t n, double *coef) {
    std::vector<double> M((size_t)n, 0.0), diag((size_t)n, 0.0), rhs((size_t)n, 0.0);
    for (int32_t k = 1; k < n - 1; k++) {
        diag[(size_t)k] = 4.0;
        rhs[(size_t)k] = 6.0 * (y[k + 1] - 2.0 * y[k] + y[k - 1]);
    }
    for (int32_t k = 2; k < n - 1; k++) {
        const double f = 1.0 / diag[(size_t)k - 1];
        diag[(size_t)k] -= f;
        rhs[(size_t)k] -= f * rhs[(size_t)k - 1];
    }
    for (int32_t k = n - 2; k >= 1; k--) {
        const double up = (k + 1 < n - 1) ? M[(size_t)k + 1] : 0.0;
        M[(size_t)k] = (rhs[(size_t)k] - up) / diag[(size_t)k];
    }
    for (int32_t k = 0; k < n - 1; k++) {
        double *c = coef + 4 * (size_t)k;
        c[0] = y[k];
        c[1] = (y[k + 1] - y[k]) - (2.0 * M[(size_t)k] + M[(size_t)k + 1]) / 6.0;
        c[2] = 0.5 * M[(size_t)k];
        c[3] = (M[(size_t)k + 1] - M[(size_t)k]) / 6.0;
    }
}

// Every pair of the complete graph on n blocks goes to one of its two ends; column j takes at most
// cap[j] = 4 m_j - 1 pairs beside its own block, with sum_j m_j items in all. m_j is the same for every
// column but for one more in the first few, and any k columns can hold their k (k - 1) / 2 inner pairs,
// so an assignment exists. Pairs are placed by increasing cyclic distance d at the column d before
// (so that a column's rows are mostly consecutive), else at the other end, else by moving pairs along a
// path of full columns to one with room.
std::vector<std::vector<int>> nao_block_pairs(int n) {
    const int total = std::max(n, (n * (n + 1) / 2 + 3) / 4);
    const int m = total / n, more = total - m * n;
    std::vector<int> room(n);
    for (int j = 0; j < n; j++) room[j] = 4 * (m + (j < more ? 1 : 0)) - 1;
    std::vector<int> owner((size_t)n * n, -1);  // of the pair {a, b}: at both (a, b) and (b, a)
    auto give = [&](int a, int b, int to) { owner[(size_t)a * n + b] = owner[(size_t)b * n + a] = to; };
    for (int d = 1; d <= n / 2; d++)
        for (int j = 0; j < n; j++) {
            const int o = (j + d) % n;
            if (owner[(size_t)j * n + o] >= 0) continue;  // n even, d = n / 2: the pair's other end came first
            // a column with room that j or o reaches by moving pairs: breadth first
            std::vector<int> from(n, -2), queue;
            int end = -1;
            for (int x : {j, o}) {
                if (from[x] != -2) continue;
                from[x] = -1;
                queue.push_back(x);
            }
            for (size_t h = 0; h < queue.size() && end < 0; h++) {
                const int x = queue[h];
                if (room[x] > 0) {
                    end = x;
                    break;
                }
                for (int y = 0; y < n; y++)
                    if (y != x && from[y] == -2 && owner[(size_t)x * n + y] == x) {  // x could pass {x, y} to y
                        from[y] = x;
                        queue.push_back(y);
                    }
            }
            if (end < 0) end = j;  // cannot happen (see above); the column then takes one item more
            room[end]--;
            int x = end;
            while (from[x] >= 0) {
                give(from[x], x, x);
                x = from[x];
            }
            give(j, o, x);
        }
    std::vector<std::vector<int>> rows(n);
    for (int j = 0; j < n; j++)
        for (int d = 0; d < n; d++) {
            const int o = (j + d) % n;
            if (d == 0 || owner[(size_t)j * n + o] == j) rows[j].push_back(o);
        }
    return rows;
}

void nao_split_h_items(int32_t b, int P, int N, int TN, int S, std::vector<HTask> &out, BlockPairs &kept, int F) {
    const int nseg = nao_split_h_nseg(P, S, F);
    auto add = [&](int j, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3) {
        for (int q = 0; q < nseg; q++)
            out.push_back({b, (uint32_t)j | (uint32_t)q << 16, r0 | r1 << 16, r2 | r3 << 16});
    };
    const int nr = (N + 31) / 32;
    if (TN != 32) {
        const int nJ = (N + TN - 1) / TN;
        for (int I = 0; 128 * I < N; I++)
            for (int J = (I * 128) / TN; J < nJ; J++) {
                uint32_t r[4];
                for (int x = 0; x < 4; x++) r[x] = 4 * I + x < nr ? (uint32_t)(4 * I + x) : kNoRows;
                add(J, r[0], r[1], r[2], r[3]);
            }
        return;
    }
    auto it = kept.find(nr);
    if (it == kept.end()) it = kept.emplace(nr, nao_block_pairs(nr)).first;
    for (int j = 0; j < nr; j++) {
        const std::vector<int> &rows = it->second[j];
        for (size_t k = 0; k < rows.size(); k += 4) {
            uint32_t r[4];
            for (size_t x = 0; x < 4; x++) r[x] = k + x < rows.size() ? (uint32_t)rows[k + x] : kNoRows;
            add(j, r[0], r[1], r[2], r[3]);
        }
    }
}
