// Host run of the fixed-point pair law (hg_pair64.cuh).  Reads from stdin
// "eps n" and then, for particle i (x v a) and each of n particles j (m x v a),
// the values as hexadecimal floats; prints the nine sums over j and the
// potential sum.  Repeats until the input ends.
#include <stdio.h>

#include "hg_pair64.cuh"

int main()
{
    double eps;
    int n;
    while (scanf("%la %d", &eps, &n) == 2) {
        double i[9], m, j[9];
        for (double &x : i)
            if (scanf("%la", &x) != 1) return 1;
        const hg::p64::Body b{i[0], i[1], i[2], i[3], i[4], i[5], i[6], i[7], i[8]};
        const hg::p64::Soft soft = hg::p64::soft(eps * eps);
        hg::p64::Sums s;
        hg::p64::Potential p;
        hg::p64::clear(s);
        hg::p64::clear(p);
        for (int k = 0; k < n; ++k) {
            if (scanf("%la", &m) != 1) return 1;
            for (double &x : j)
                if (scanf("%la", &x) != 1) return 1;
            if (eps > 0.0)
                hg::p64::pair<false>(b, j[0], j[1], j[2], m, j[3], j[4], j[5], j[6], j[7], j[8], soft, s);
            else
                hg::p64::pair<true>(b, j[0], j[1], j[2], m, j[3], j[4], j[5], j[6], j[7], j[8], soft, s);
            hg::p64::count_pair(s);
            hg::p64::Limbs ml;
            uint32_t low = 0;
            const int em = hg::p64::mass_limbs(m, ml, low);
            const bool self = j[0] == i[0] && j[1] == i[1] && j[2] == i[2];
            hg::p64::pair_potential(j[0] - i[0], j[1] - i[1], j[2] - i[2], ml, em, self, soft, p);
            if (k % hg::p64::kFold64 == hg::p64::kFold64 - 1) hg::p64::fold_fp64(p);
        }
        hg::p64::finish(s);
        hg::p64::fold_fp64(p);
        for (double x : s.s) printf("%a ", x);
        printf("%a\n", p.s);
    }
    return 0;
}
