// Host-side check of a server's account of the resident kernel's layouts
// (lpb_serve.cu): they are charged to the memory budget, are not made where it
// has no room (the step kernels run), and give way to a request that needs
// their room.  Runs on the stand-in runtime, whose LPs never finish.  Prints
// "ok" or the first failure.
#include <chrono>
#include <cstdio>
#include <thread>
#include <vector>

#include "fake_cuda.h"
#include "lpb_engine.h"
#include "lpb_serve.h"

static int fail_at(const char* what, long long v) {
    std::printf("%s (%lld)\n", what, v);
    return 1;
}

static lpb_handle make(int m, int n) {
    std::vector<int64_t> rp(m + 1);
    std::vector<int32_t> ci;
    std::vector<double> v, cost(n, 1.0), lo(m, -1.0), hi(m, 1.0), xl(n, 0.0), xu(n, 1.0);
    for (int i = 0; i < m; ++i) {
        for (int k = 0; k < 3; ++k) ci.push_back((i + k) % n), v.push_back(1.0 + k);
        rp[i + 1] = (int64_t)ci.size();
    }
    lpb_handle h = nullptr;
    return lpb_create(m, n, rp[m], rp.data(), ci.data(), v.data(), cost.data(), lo.data(), hi.data(), xl.data(), xu.data(),
                      nullptr, &h) == LPB_OK
               ? h
               : nullptr;
}

template <typename F>
static bool within_5s(F f) {
    for (int k = 0; k < 5000; ++k) {
        if (f()) return true;
        std::this_thread::sleep_for(std::chrono::milliseconds(1));
    }
    return false;
}

static int64_t used(lpb_server_t s) {
    lpb_server_stats st{};
    lpb_server_stats_get(s, &st);
    return st.hbm_used_bytes;
}
static int state(lpb_server_t s, int64_t id) {
    lpb_request_info q{};
    lpb_server_request_info(s, id, &q);
    return q.state;
}

int main() {
    // every admitted LP is running (its record says so), at any number of LPs
    fake::on_read = [](void* d, size_t n) {
        if (n % sizeof(lpb::ColRecord) != 0 || n > 16 * sizeof(lpb::ColRecord)) return;
        for (size_t k = 0; k < n / sizeof(lpb::ColRecord); ++k) ((lpb::ColRecord*)d)[k].status = -1;
    };
    static_assert(sizeof(lpb::Control) % sizeof(lpb::ColRecord) != 0, "the copies are told apart by their size");
    const int m = 200, n = 400, cols = 32;
    lpb_server_options o;
    lpb_server_default_options(&o);
    o.lane_columns = cols;
    o.max_groups = 1 + 2;
    int64_t lanes = 0, layout = 0;
    std::vector<lpb_lp_spec> sp(cols, lpb_lp_spec{0, -1, 0.0, 0.0, 1.0});
    lpb_request q{};
    q.matrix_id = 0;
    q.specs = sp.data();
    q.tol = 1e-4;
    q.max_iter = 1 << 30;
    q.warm_request = -1;
    const int64_t each = ((int64_t)n + m) * 8 + (int64_t)sizeof(lpb_lp_spec);  // footprint of a request's LP
    for (int round = 0; round < 3; ++round) {
        // round 0: room for everything; 1: none for a layout; 2: for a layout or a second request
        lpb_handle h = make(m, n);
        if (!h) return fail_at("create", round);
        o.hbm_budget_bytes = round == 0 ? (int64_t)1 << 34 : round == 1 ? lanes + each + layout - 1 : lanes + each + layout;
        lpb_server_t s = nullptr;
        int32_t id = -1;
        if (lpb_server_create(&o, &s) != LPB_OK || lpb_server_attach(s, h, &id) != LPB_OK) return fail_at("attach", round);
        if (round == 0) lanes = used(s);
        if (used(s) != lanes) return fail_at("lanes", used(s));
        const long steps = fake::launches("k_step"), res = fake::launches("k_resident");
        int64_t first = -1, second = -1;
        q.num_lps = 1;
        if (lpb_server_submit(s, &q, &first) != LPB_OK) return fail_at("submit", round);
        if (!within_5s([&] { return fake::launches("k_step") > steps + 1000 || fake::launches("k_resident") > res + 10; }))
            return fail_at("no interval runs", round);
        if (round == 1) {
            if (fake::launches("k_resident") != res) return fail_at("a layout without room", round);
            if (used(s) != lanes + each) return fail_at("account without a layout", used(s) - lanes - each);
        } else {
            if (fake::launches("k_step") != steps) return fail_at("steps beside a layout", round);
            if (round == 0) layout = used(s) - lanes - each;
            if (layout <= 0 || used(s) != lanes + each + layout) return fail_at("account of a layout", used(s) - lanes - each);
        }
        if (round == 2) {
            q.num_lps = (int32_t)(layout / each);
            if (q.num_lps < 1 || q.num_lps + 1 > cols) return fail_at("the second request's size", q.num_lps);
            if (lpb_server_submit(s, &q, &second) != LPB_OK) return fail_at("submit", round);
            if (!within_5s([&] { return state(s, second) == 1; })) return fail_at("a request waits for a layout's room", state(s, second));
            if (!within_5s([&] { return fake::launches("k_step") > steps + 1000; })) return fail_at("no steps without the layout", round);
            if (used(s) != lanes + each * (1 + q.num_lps)) return fail_at("account after the layout", used(s) - lanes);
        }
        if (used(s) > o.hbm_budget_bytes) return fail_at("over budget", used(s));
        lpb_server_destroy(s);
        if (h->res_charge) return fail_at("the account outlives its server", round);
        // a layout made for one server is not on the next one's account
        o.hbm_budget_bytes = (int64_t)1 << 34;
        if (lpb_server_create(&o, &s) != LPB_OK || lpb_server_attach(s, h, &id) != LPB_OK) return fail_at("second server", round);
        lpb_tuning t{64, 64, 0, 0};
        if (lpb_set_tuning(h, &t) != LPB_OK || used(s) != lanes) return fail_at("account of the second server", used(s) - lanes);
        lpb_server_destroy(s);
        lpb_destroy(h);
        if (fake::live_bytes() != 0) return fail_at("memory left", (long long)fake::live_bytes());
    }
    std::printf("ok\n");
    return 0;
}
