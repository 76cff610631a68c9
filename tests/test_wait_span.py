"""Timeouts of the server's blocking calls (csrc/wait_span.cuh), run on the host: the
deadline that a condition variable waits for is never before now."""
from test_list_rules import run


def test_deadlines(tmp_path):
    run(tmp_path, """
#include "wait_span.cuh"
#include <cmath>
#include <condition_variable>
#include <limits>
#include <mutex>
int main() {
    using D = std::numeric_limits<double>;
    const auto now = std::chrono::steady_clock::now();
    double last = -1.0;
    for (double ms : {0.0, 1e-7, 1e-3, 0.5, 1.0, 3e5, 1e9, 3e10, 4e10, 9.3e12, 1e18, D::max(), D::infinity()}) {
        const auto d = wait_span(ms);
        CHECK(d.count() >= 0 && now + d >= now);
        const double got = std::chrono::duration<double, std::milli>(d).count();
        CHECK(got >= last);
        if (ms <= 3e10) CHECK(std::fabs(got - ms) <= 1e-6 + 1e-12 * ms);
        if (ms > 3e10) CHECK(got > 3e10);
        last = got;
    }
    for (double ms : {-1.0, -D::infinity(), D::quiet_NaN()}) CHECK(wait_span(ms).count() == 0);
    // a wait without end waits: the predicate is looked at again when it is told to
    std::mutex m;
    std::condition_variable cv;
    std::unique_lock<std::mutex> lk(m);
    int looks = 0;
    CHECK(cv.wait_for(lk, wait_span(D::infinity()), [&] { return ++looks >= 1; }));
    CHECK(!cv.wait_for(lk, wait_span(1.0), [] { return false; }));
    return 0;
}
""")
