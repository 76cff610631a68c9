"""The index rules of the tile lists (csrc/list_rules.cuh), run on the host: whatever a
depth order holds after a wait between CTAs ran out, the list kernels index only their
own view's tiles.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2505_22335_gb300", "csrc")


def run(tmp_path, body):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src = tmp_path / "t.cpp"
    src.write_text('#include "list_rules.cuh"\n#include <algorithm>\n#include <cstdio>\n#include <random>\n'
                   '#include <vector>\nusing namespace ups;\n'
                   '#define CHECK(c) do { if (!(c)) { std::printf("%s\\n", #c); return 1; } } while (0)\n' + body)
    exe = str(tmp_path / "t")
    subprocess.run([cxx, "-std=c++17", "-O1", "-fsanitize=undefined", "-fno-sanitize-recover", "-I", CSRC, str(src), "-o", exe],
                   check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr


def test_ids_of_a_view(tmp_path):
    run(tmp_path, """
int main() {
    std::mt19937 rng(1);
    // (Gaussians a view, views): small, and up to 2^31 Gaussian-views
    const uint32_t cases[][2] = {{1, 1}, {1, 64}, {7, 3}, {4096, 2}, {2147483647u, 1}, {715827882u, 3}, {33554431u, 64}};
    for (auto &c : cases) {
        const uint32_t N = c[0], V = c[1];
        for (uint32_t v = 0; v < V; ++v) {
            const uint64_t lo = (uint64_t)v * N, hi = lo + N;
            uint32_t ids[] = {0u, (uint32_t)lo - 1u, (uint32_t)lo, (uint32_t)(lo + N / 2), (uint32_t)hi - 1u,
                              (uint32_t)hi, N * V - 1u, N * V, 0x7fffffffu, 0x80000000u, 0xffffffffu};
            for (uint32_t id : ids) CHECK(of_view(id, v, N) == (id >= lo && id < hi));
            for (int i = 0; i < 200; ++i) {
                const uint32_t id = rng();
                CHECK(of_view(id, v, N) == (id >= lo && id < hi));
            }
        }
    }
    // pyramid levels of unequal size: a Gaussian's column lies in its own view's tiles, and
    // whatever the order holds, a run only indexes the tiles of the view it counts
    const int tiles[3] = {1200, 300, 80}, N = 500, V = 3;
    std::vector<int> tile(N * V);
    for (int i = 0; i < N * V; ++i) tile[i] = rng() % tiles[i / N];
    for (int trial = 0; trial < 50; ++trial) {
        std::vector<uint32_t> order(N * V);
        for (auto &o : order) o = rng() % 4 ? rng() % (N * V) : rng();
        for (int v = 0; v < V; ++v)
            for (int i = 0; i < N; ++i) {
                const uint32_t id = order[v * N + i];
                if (of_view(id, v, N)) CHECK(tile[id] < tiles[v]);
            }
    }
    return 0;
}
""")


def test_list_positions_stay_in_the_buffer(tmp_path):
    # The arithmetic of bin.cu (counts a run, their prefix, ranges, fill) over orders that
    # repeat ids: every position that the rules let through lies in the buffer, and of a
    # sound order every entry is kept.
    run(tmp_path, """
template <bool CAPPED> int fill(const std::vector<uint32_t> &order, const std::vector<std::vector<int>> &tiles_of,
                                int tiles, uint32_t cap, uint32_t n, bool sound) {
    const int N = (int)order.size(), R = 64, nb = (N + R - 1) / R;
    std::vector<uint32_t> cnt((size_t)nb * tiles), tot(tiles), list(n, ~0u);
    for (int i = 0; i < N; ++i)
        if (of_view(order[i], 0, N))
            for (int t : tiles_of[order[i]]) cnt[(size_t)(i / R) * tiles + t]++;
    for (int t = 0; t < tiles; ++t)
        for (int b = 0; b < nb; ++b) {
            const uint32_t c = cnt[(size_t)b * tiles + t];
            cnt[(size_t)b * tiles + t] = tot[t];
            tot[t] += c;
        }
    std::vector<std::pair<uint32_t, uint32_t>> rg(tiles);
    uint32_t at = 0, kept = 0;
    for (int t = 0; t < tiles; ++t) {
        const uint32_t k = std::min(tot[t], cap);
        rg[t] = {std::min(at, n), std::min(at + k, n)};
        at += k;
    }
    for (int b = 0; b < nb; ++b) {
        std::vector<Slot<CAPPED>> slot(tiles);
        for (int t = 0; t < tiles; ++t) {
            slot[t].next = rg[t].first + std::min(cnt[(size_t)b * tiles + t], rg[t].second - rg[t].first);
            if constexpr (CAPPED) slot[t].stop = rg[t].second;
        }
        for (int i = b * R; i < std::min(N, (b + 1) * R); ++i) {
            if (!of_view(order[i], 0, N)) continue;
            for (int t : tiles_of[order[i]]) {
                const uint32_t pos = slot[t].next++;
                if (!slot[t].fits(pos, n)) continue;
                CHECK(pos < list.size());
                list[pos] = order[i];
                ++kept;
            }
        }
    }
    if (sound) CHECK(kept == std::min(at, n));
    return 0;
}

int main() {
    std::mt19937 rng(2);
    for (int trial = 0; trial < 60; ++trial) {
        const int N = 1 + rng() % 700, tiles = 1 + rng() % 40;
        std::vector<std::vector<int>> tiles_of(N);
        uint32_t n = 0;
        for (auto &t : tiles_of) {
            for (int k = rng() % 4; k > 0; --k) t.push_back(rng() % tiles);
            n += (uint32_t)t.size();
        }
        std::vector<uint32_t> order(N);
        for (int i = 0; i < N; ++i) order[i] = i;
        std::shuffle(order.begin(), order.end(), rng);
        uint32_t most = 0;  // the id with the most tiles: repeated, more entries than the buffer has
        for (int i = 0; i < N; ++i)
            if (tiles_of[i].size() > tiles_of[most].size()) most = i;
        for (int broken = 0; broken < 2; ++broken) {
            if (broken)
                for (int i = 0; i < N; ++i)
                    if (rng() % 3 == 0) order[i] = rng() % 4 ? most : rng();
            if (fill<false>(order, tiles_of, tiles, ~0u, n, !broken)) return 1;
            for (uint32_t cap : {1u, 7u, 1000u})
                if (fill<true>(order, tiles_of, tiles, cap, n, !broken)) return 1;
        }
    }
    return 0;
}
""")
