// Host-side check of an admission's cost: LPs that are infeasible from their
// overrides alone end at once, in as many calls of the runtime whether they are
// eight or a thousand.  Runs on the stand-in runtime, where every LP ends so.
// Prints "ok" or the first failure.
#include <cstdio>
#include <vector>

#include "fake_cuda.h"
#include "lpb.h"

int main() {
    const int m = 20, n = 30;
    std::vector<int64_t> rp(m + 1);
    std::vector<int32_t> ci;
    std::vector<double> v, cost(n, 1.0), lo(m, -1.0), hi(m, 1.0), xl(n, 0.0), xu(n, 1.0);
    for (int i = 0; i < m; ++i) {
        ci.push_back(i);
        v.push_back(1.0);
        rp[i + 1] = (int64_t)ci.size();
    }
    lpb_handle h = nullptr;
    if (lpb_create(m, n, rp[m], rp.data(), ci.data(), v.data(), cost.data(), lo.data(), hi.data(), xl.data(), xu.data(),
                   nullptr, &h) != LPB_OK)
        return std::printf("create\n"), 1;
    std::vector<lpb_lp_spec> sp(1000, lpb_lp_spec{1, 3, 5.0, 4.0, 1.0});
    long calls[2] = {0, 0};
    const int lps[2] = {1000, 8};  // the wider batch first: the lane's own memory is there for the second
    for (int k = 0; k < 2; ++k) {
        lpb_batch_t b = nullptr;
        long before = 0;
        for (int again = 0; again < 2; ++again) {
            before = fake::memsets() + fake::launches("");
            if (lpb_solve(h, lps[k], sp.data(), 1e-4, 64, nullptr, nullptr, &b) != LPB_OK) return std::printf("solve\n"), 1;
            lpb_batch_free(b);
        }
        calls[k] = fake::memsets() + fake::launches("") - before;
    }
    if (calls[0] != calls[1]) return std::printf("calls for 1000 and 8 LPs: %ld and %ld\n", calls[0], calls[1]), 1;
    lpb_destroy(h);
    std::printf("ok\n");
    return 0;
}
