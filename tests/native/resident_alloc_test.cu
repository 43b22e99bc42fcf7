// Host-side check of the resident kernel's layouts (lpb_resident.cu) when the
// device has no memory for them: the choice of the kernel is no error then, the
// step kernels run, nothing of the layout is left behind and no second try
// adds to it.  And of what making one costs the device's other users: nothing
// waits for the whole device, and a batch that the step kernels run faster
// allocates nothing.  Runs on the stand-in runtime.  Prints "ok" or the first failure.
#include <cstdio>
#include <vector>

#include "fake_cuda.h"
#include "lpb_engine.h"

static int fail_at(const char* what, long k) {
    std::printf("%s (%ld)\n", what, k);
    return 1;
}

static lpb_handle make(int m, int n, int each, int precision) {
    std::vector<int64_t> rp(m + 1);
    std::vector<int32_t> ci;
    std::vector<double> v, cost(n, 1.0), lo(m, -1.0), hi(m, 1.0), xl(n, 0.0), xu(n, 1.0);
    for (int i = 0; i < m; ++i) {
        for (int k = 0; k < each; ++k) ci.push_back((i + k) % n), v.push_back(1.0 + k);
        rp[i + 1] = (int64_t)ci.size();
    }
    lpb_options o;
    lpb_default_options(&o);
    o.precision = precision;
    lpb_handle h = nullptr;
    return lpb_create(m, n, rp[m], rp.data(), ci.data(), v.data(), cost.data(), lo.data(), hi.data(), xl.data(), xu.data(), &o,
                      &h) == LPB_OK
               ? h
               : nullptr;
}

int main() {
    using namespace lpb;
    bool done = false;
    for (long k = 0; !done; ++k) {
        lpb_handle h = make(200, 400, 3, LPB_MIXED);
        if (!h) return fail_at("create", k);
        Lane& ln = h->lane[kPrecF32];
        if (lane_reserve(h, ln, kPrecF32, 16, 1) != LPB_OK || ensure_check_ws(h, ln.cap) != LPB_OK) return fail_at("lane", k);
        ln.ncol = 16;
        ln.col_group.assign(ln.cap, 0);
        const size_t before = fake::live_bytes();
        const long waits = fake::device_waits();
        for (int again = 0; again < 3; ++again) {
            ResShape shape;
            ResPlan* plan = nullptr;
            Lane* lp = &ln;
            if (again == 0) fake::fail_after(k, 1 << 20);
            if (res_choose<float>(&h, &lp, 1, &shape, &plan) != LPB_OK) return fail_at("no memory for a layout ends the solve", k);
            if (again == 0) {
                fake::fail_none();
                done = shape.C > 0;
            }
            if (done != (shape.C > 0)) return fail_at("the choice changes", k);
            if (h->res_plans.size() != 1) return fail_at("entries for one layout", (long)h->res_plans.size());
            if (!done && fake::live_bytes() != before) return fail_at("memory of a layout that is not used", k);
            if (fake::device_waits() != waits) return fail_at("a wait for the whole device", fake::device_waits() - waits);
            if (fake::last_error()) return fail_at("an error is left for the next launch", k);
        }
        const long steps = fake::launches("k_step"), res = fake::launches("k_resident");
        if (lane_interval<float>(h, ln, 64, 0, h->stream, nullptr) != LPB_OK) return fail_at("interval", k);
        if (done ? fake::launches("k_resident") != res + 1 : fake::launches("k_step") != steps + 128)
            return fail_at("kernels of the interval", k);
        ln.ncol = 0;
        lpb_destroy(h);
        if (fake::live_bytes() != 0) return fail_at("memory left", k);
    }
    // 30,000 entries in FP64: the step kernels' case
    lpb_handle h = make(1000, 2000, 30, LPB_FP64);
    if (!h) return fail_at("create", -1);
    Lane& ln = h->lane[kPrecF64];
    if (lane_reserve(h, ln, kPrecF64, 2, 1) != LPB_OK || ensure_check_ws(h, ln.cap) != LPB_OK) return fail_at("lane", -1);
    ln.ncol = 2;
    const size_t before = fake::live_bytes();
    ResShape shape;
    ResPlan* plan = nullptr;
    Lane* lp = &ln;
    if (res_choose<double>(&h, &lp, 1, &shape, &plan) != LPB_OK || shape.C != 0) return fail_at("the choice", shape.C);
    if (fake::live_bytes() != before) return fail_at("memory of a layout that is not used", -1);
    ln.ncol = 0;
    lpb_destroy(h);
    std::printf("ok\n");
    return 0;
}
