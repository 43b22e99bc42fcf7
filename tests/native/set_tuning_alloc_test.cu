// Host-side check of a threshold change that runs out of memory
// (lpb_set_tuning): whichever of its allocations fails, the handle keeps a
// complete list of rows -- the old threshold's where it can be had again --
// and a handle whose rows could not be laid out at all refuses to solve
// until a threshold change succeeds.  Runs on the stand-in runtime.  Prints
// "ok" or the first failure.
#include <cstdio>
#include <vector>

#include "fake_cuda.h"
#include "lpb_engine.h"
#include "lpb_serve.h"

static int fail_at(const char* what, long k) {
    std::printf("%s (allocation %ld)\n", what, k);
    return 1;
}

static bool whole(const lpb::Csr& c) {
    return c.long_thr > 0 && c.n_short == c.rows - c.n_long && c.srec && c.nrec && c.pci;
}

int main() {
    const int m = 300, n = 200;
    std::vector<int64_t> rp(m + 1);
    std::vector<int32_t> ci;
    std::vector<double> v, cost(n, 1.0), lo(m, -1.0), hi(m, 1.0), xl(n, 0.0), xu(n, 1.0);
    for (int i = 0; i < m; ++i) {
        for (int k = 0; k < 3; ++k) ci.push_back((i + 7 * k) % n), v.push_back(1.0 + k);
        rp[i + 1] = (int64_t)ci.size();
    }
    lpb_options o;
    lpb_default_options(&o);
    lpb_lp_spec sp{0, -1, 0.0, 0.0, 1.0};
    // one allocation of a threshold change fails, the k-th: until none does
    bool done = false;
    for (long k = 0; !done; ++k) {
        lpb_handle h = nullptr;
        if (lpb_create(m, n, rp[m], rp.data(), ci.data(), v.data(), cost.data(), lo.data(), hi.data(), xl.data(), xu.data(),
                       &o, &h) != LPB_OK)
            return fail_at("create", k);
        if (!whole(h->A) || !whole(h->At)) return fail_at("rows of a new handle", k);
        const int epoch = h->ws_epoch;
        const int p = h->At.long_thr, d = h->A.long_thr;
        lpb_tuning t{16, 64, 0, 0};
        fake::fail_after(k, 1);
        const lpb_err rc = lpb_set_tuning(h, &t);
        fake::fail_none();
        done = rc == LPB_OK;
        if (done && (h->At.long_thr != 16 || h->A.long_thr != 64)) return fail_at("thresholds after the change", k);
        if (!done) {
            if (rc != LPB_ERR_OOM) return fail_at("error code", k);
            if (h->At.long_thr != p && h->At.long_thr != 16) return fail_at("primal threshold after a failure", k);
            if (h->A.long_thr != d) return fail_at("dual threshold after a failure", k);
            if (h->ws_epoch == epoch) return fail_at("captured intervals outlive freed rows", k);
        }
        if (!whole(h->A) || !whole(h->At)) return fail_at("rows after a failure", k);
        if (lpb_set_tuning(h, &t) != LPB_OK || h->At.long_thr != 16 || h->A.long_thr != 64) return fail_at("second try", k);
        if (!whole(h->A) || !whole(h->At)) return fail_at("rows after the second try", k);
        lpb_destroy(h);
        if (fake::live_bytes() != 0) return fail_at("memory left", k);
    }
    // all allocations fail from the k-th on
    done = false;
    for (long k = 0; !done; ++k) {
        lpb_handle h = nullptr;
        if (lpb_create(m, n, rp[m], rp.data(), ci.data(), v.data(), cost.data(), lo.data(), hi.data(), xl.data(), xu.data(),
                       &o, &h) != LPB_OK)
            return fail_at("create", k);
        lpb_tuning t{16, 64, 0, 0};
        fake::fail_after(k, 1 << 20);
        done = lpb_set_tuning(h, &t) == LPB_OK;
        fake::fail_none();
        if (!whole(h->A) || !whole(h->At)) {
            const long steps = fake::launches("k_step") + fake::launches("k_resident");
            lpb_batch_t b = nullptr;
            lpb_tuning got{};
            if (lpb_solve(h, 1, &sp, 1e-4, 64, nullptr, nullptr, &b) == LPB_OK || b) return fail_at("a solve without rows", k);
            const lpb_lp_spec* sps[] = {&sp};
            const int32_t one = 1;
            if (lpb_solve_multi(1, &h, &one, sps, 1e-4, 64, &b) == LPB_OK) return fail_at("a joint solve without rows", k);
            if (lpb_solve_dev(h, 1, &sp, 1e-4, 64, nullptr, nullptr, &b) == LPB_OK) return fail_at("a device solve without rows", k);
            const int32_t width = 4;
            double us = 0.0;
            if (lpb_tune_batch(h, &width, 1, &us, nullptr) == LPB_OK) return fail_at("steps timed without rows", k);
            lpb_server_t srv = nullptr;
            int32_t id = -1;
            if (lpb_server_create(nullptr, &srv) != LPB_OK) return fail_at("server", k);
            if (lpb_server_attach(srv, h, &id) == LPB_OK) return fail_at("a matrix served without rows", k);
            lpb_server_destroy(srv);
            if (steps != fake::launches("k_step") + fake::launches("k_resident")) return fail_at("steps run without rows", k);
            if (lpb_get_tuning(h, &got) != LPB_OK) return fail_at("tuning without rows", k);
        }
        if (lpb_set_tuning(h, &t) != LPB_OK || h->At.long_thr != 16 || h->A.long_thr != 64 || !whole(h->A) || !whole(h->At))
            return fail_at("second try after no memory at all", k);
        lpb_destroy(h);
        if (fake::live_bytes() != 0) return fail_at("memory left", k);
    }
    std::printf("ok\n");
    return 0;
}
