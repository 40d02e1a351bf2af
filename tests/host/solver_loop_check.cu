// Host-side check of the solver's device-driven loop (compiled with nvcc as a
// host program; no GPU needed): segments end after the set number of
// iterations, or with the solve, whatever values the graph's handles have.
#include <cstdio>

#include "tm_cg.cuh"

using namespace twm;

int main()
{
    int bad = 0;
    const unsigned long long handles[] = {0, 1, ~0ull};
    for (unsigned long long h : handles)
        for (int n : {1, 2, 50})
            for (int last : {1, 7, 1000}) {   // the iteration that ends the solve
                CgScalars s{};
                if (s.has_loop || s.has_update) ++bad;   // no graph: no conditional node is touched
                s.set_graph(h, h != 1, h, n);
                if (!s.has_loop || s.has_update != (h != 1)) ++bad;
                int done = 0;
                for (int segment = 0; segment < 3 && !s.done; ++segment) {
                    int k = 0;
                    bool more = true;
                    while (more && k < 2000) {
                        ++k;
                        s.done = ++done >= last;
                        more = cg_loop_more(&s);
                    }
                    if (k != (s.done ? (last - 1) % n + 1 : n)) ++bad;
                }
            }
    printf("%d failures\n", bad);
    return bad != 0;
}
