// Where the entries of K's rows go in the dense blocks of the prefactorisation (host and device).
#pragma once

#ifdef __CUDACC__
#define PDG_ROWS_HD __host__ __device__ __forceinline__
#else
#define PDG_ROWS_HD inline
#endif

namespace pdg {

// position of `c` in the ascending list col[lo, hi), or -1
PDG_ROWS_HD int find_col(const int* col, int lo, int hi, int c) {
    const int end = hi;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (col[mid] < c) lo = mid + 1;
        else hi = mid;
    }
    return lo < end && col[lo] == c ? lo : -1;
}

// Column c of a row of a domain's internal vertices (`count` from `first` on; its interface vertices are
// bnd[bnd_first, bnd_first + bnd_count), ascending, numbered from n_int on): the column of K_ii, or count + the column
// of K_ib, or -1 when the domain has no place for it (another domain's internal vertex, or an interface vertex that
// is not on its list).
PDG_ROWS_HD int domain_place(int c, int first, int count, const int* bnd, int bnd_first, int bnd_count, int n_int) {
    if (c >= first && c < first + count) return c - first;
    if (c < n_int) return -1;
    const int p = find_col(bnd, bnd_first, bnd_first + bnd_count, c - n_int);
    return p < 0 ? -1 : count + p - bnd_first;
}

}  // namespace pdg
