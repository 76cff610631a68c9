"""Who is told of a wait that ran out on the GPU (csrc/lost_wait.cuh), run on the host: the
batch whose kernels lost it, and no later one.
"""
import os

from test_list_rules import CSRC, run


def test_the_batch_that_lost_a_wait_fails(tmp_path, monkeypatch):
    monkeypatch.setenv("CPLUS_INCLUDE_PATH", os.path.join(os.path.dirname(os.path.dirname(CSRC)), "include"))
    run(tmp_path, """
#include "lost_wait.cuh"
int main() {
    // a slot: a forward takes the word after its projection (what launches before left), the
    // end of the batch takes it once more.  Batch b of 6 loses a wait before its forward's
    // check (2), after it (1), or not at all (0).
    int word = 0;
    const LostWait slot{&word};
    for (int mask = 0; mask < 729; ++mask) {
        int m = mask;
        for (int b = 0; b < 6; ++b, m /= 3) {
            const int loses = m % 3;
            std::vector<int> reqs = {UPS_PENDING, UPS_ERR_CANCELLED, UPS_PENDING};
            if (loses == 2) word = 1;
            const bool early = slot.take();  // the forward fails its own batch
            CHECK(early == (loses == 2));
            if (loses == 1) word = 1;
            if (!early) {
                const bool lost = slot.take();
                for (int &r : reqs) r = settled_status(r, lost);
                CHECK(reqs[0] == (loses ? UPS_ERR_TIMEOUT : UPS_OK) && reqs[2] == reqs[0]);
                CHECK(reqs[1] == UPS_ERR_CANCELLED);
            }
            CHECK(word == 0 && !slot.take());
        }
    }
    CHECK(!LostWait{}.take());
    return 0;
}
""")
