// Every order of the warps of a CTA of the 2D FP64 sweep that its waits (csrc/sweep2d_f64_waits.h) allow, for a band of
// PR units of RPW rows, NC velocity groups and M moment warps on n1 columns, with blocks of B columns instead of 16.
// Sweeping, record and moment warps take small steps (a wait that is fulfilled and the reads and writes behind it, then
// the release); what a step reads is checked when it begins and when it ends.  The band below is always there.
// Usage: model PR NC RPW n1 M with_group_wait -> "ok STATES" or "violation WHAT".
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <deque>
#include <string>
#include <unordered_set>

#include "sweep2d_f64_waits.h"

using namespace dvm::f64waits;

// (the bound of a wait of the test hook may be as large as its type allows)
static_assert(inner_bound(2000000000LL) == 128000000000LL && inner_bound(1) == 64, "64 times the bound");
static_assert(inner_bound(0x7fffffffffffffffLL) == 0x7fffffffffffffffLL && inner_bound(1LL << 58) > (1LL << 62), "no overflow");

namespace {

constexpr int B = 3;   // (a record block is written while the sweep is inside the block before it: B > RPW)
int PR, NC, RPW, N1, M, W, NBLK, STEPS;
bool GROUP_WAIT;
const char* broken = nullptr;

struct Sweep { unsigned char col, busy; };                        // steps finished; a step is under way
struct Mom { unsigned char kb, w, phase, last; };                 // block, sweeping warp, 0 .. 4
struct State {
    Sweep sw[6];
    Mom mo[6];
    unsigned char mom[6], rec[3], rk, rp, rbusy;                  // record warp: block, unit, writing
    unsigned char cnt[2][3], part[2][6], out[3];                  // part: block + 1; out: bits of the blocks written
};

int begun(const State& s, int w) { return s.sw[w].col + s.sw[w].busy; }

// column c of a row (0 lower, 1 upper) of warp w is in its ring of 2 B columns
bool in_ring(const State& s, int w, int row, int c) {
    const int n = std::min(begun(s, w) - row, N1);                // columns written
    return c < n && c + 2 * B >= n;
}

bool record_there(const State& s, int p, int c) {                 // of column c; not being overwritten
    const int k = c / B, written = s.rec[p] + (s.rbusy && s.rp == p ? 1 : 0);
    return k < s.rec[p] && k + 2 >= written;
}

void must(bool ok, const char* what) { if (!ok && !broken) broken = what; }

void check_step(const State& s, int w) {                          // what the step under way reads
    const int p = w / NC, c = s.sw[w].col;
    for (int e = c; e <= c + 1; ++e)
        if (e < N1) must(record_there(s, p, e), "record");
    if (c < N1)
        for (int i = 1; i <= (RPW == 2 ? 1 : 2); ++i)
            if (p >= i)
                for (int r = 0; r < RPW; ++r) must(in_ring(s, w - i * NC, r, c), "upstream row");
}

void check_sum(const State& s, const Mom& m) {
    for (int c = m.kb * B; c < std::min((m.kb + 1) * B, N1); ++c)
        for (int r = 0; r < RPW; ++r) must(in_ring(s, m.w, r, c), "summed h");
}

void check_parts(const State& s, const Mom& m) {
    const int p = m.w / NC;
    for (int g = 0; g < NC; ++g) must(s.part[m.kb & 1][p * NC + g] == m.kb + 1, "group sum");
}

bool block_ready(const State& s, int w, int k) {
    const int p = w / NC;
    if (s.rec[p] < records_of_block(k)) return false;
    if (k < 2) return true;
    if (s.mom[w] < own_moments(k)) return false;
    if (p + 1 < PR && s.sw[w + NC].col < rows_above<B>(k)) return false;
    return !(RPW == 1 && p + 2 < PR && s.sw[w + 2 * NC].col < rows_above<B>(k));
}

// the next state when agent a (sweeping warps, moment warps, record warp) takes a step; false: it waits or is done
bool advance(State& s, int a) {
    if (a < W) {
        Sweep& v = s.sw[a];
        if (v.busy) {
            check_step(s, a);
            v.busy = 0;
            ++v.col;
            return true;
        }
        if (v.col >= STEPS) return false;
        const int c = v.col, cn = c + 1;
        if (c == 0 && !block_ready(s, a, 0)) return false;
        if (cn % B == 0 && cn < N1 && !block_ready(s, a, cn / B)) return false;
        if (c < N1 && a >= NC && s.sw[a - NC].col < row_below(c, RPW)) return false;
        v.busy = 1;
        check_step(s, a);
        return true;
    }
    if (a < W + M) {
        Mom& m = s.mo[a - W];
        if (m.kb >= NBLK) return false;
        const int p = m.w / NC;
        switch (m.phase) {
        case 0:
            if (s.sw[m.w].col < swept<B>(m.kb, N1, RPW)) return false;
            check_sum(s, m);
            m.phase = 1;
            return true;
        case 1:
            if (NC > 1 && GROUP_WAIT && m.kb >= 2)
                for (int g = 0; g < NC; ++g)
                    if (s.mom[p * NC + g] < group_moments(m.kb)) return false;
            check_sum(s, m);
            s.part[m.kb & 1][m.w] = m.kb + 1;
            m.phase = 2;
            return true;
        case 2:
            m.last = s.cnt[m.kb & 1][p]++ == ((m.kb >> 1) + 1) * NC - 1;
            if (m.last) check_parts(s, m);
            m.phase = 3;
            return true;
        case 3:
            if (m.last) {
                check_parts(s, m);
                must(!(s.out[p] >> m.kb & 1), "block written twice");
                s.out[p] |= 1 << m.kb;
            }
            s.mom[m.w] = m.kb + 1;
            m.phase = m.last = 0;
            m.w += M;
            if (m.w >= W) {
                m.w = a - W;
                ++m.kb;
            }
            return true;
        }
    }
    // record warp: units in turn, block by block
    if (s.rk >= NBLK) return false;
    if (!s.rbusy) {
        for (int g = 0; s.rk >= 2 && g < NC; ++g)
            if (s.sw[s.rp * NC + g].col < record_readers<B>(s.rk, RPW)) return false;
        s.rbusy = 1;
        return true;
    }
    s.rbusy = 0;
    s.rec[s.rp] = s.rk + 1;
    if (++s.rp == PR) {
        s.rp = 0;
        ++s.rk;
    }
    return true;
}

}  // namespace

int main(int argc, char** argv) {
    if (argc != 7) return 2;
    PR = atoi(argv[1]);
    NC = atoi(argv[2]);
    RPW = atoi(argv[3]);
    N1 = atoi(argv[4]);
    M = atoi(argv[5]);
    GROUP_WAIT = atoi(argv[6]) != 0;
    W = PR * NC;
    NBLK = (N1 + B - 1) / B;
    STEPS = N1 + RPW - 1;
    if (W > 6 || PR > 3 || M > 6 || M > W || NBLK > 8) return 2;
    State s0;
    memset(&s0, 0, sizeof s0);
    for (int j = 0; j < M; ++j) s0.mo[j].w = j;
    std::unordered_set<std::string> seen;
    std::deque<State> todo{s0};
    auto key = [](const State& s) { return std::string(reinterpret_cast<const char*>(&s), sizeof s); };
    seen.insert(key(s0));
    while (!todo.empty()) {
        const State s = todo.front();
        todo.pop_front();
        bool moved = false;
        for (int a = 0; a <= W + M; ++a) {
            State t = s;
            if (!advance(t, a)) continue;
            moved = true;
            if (broken) return printf("violation %s\n", broken), 0;
            if (seen.insert(key(t)).second) todo.push_back(t);
        }
        if (moved) continue;
        for (int w = 0; w < W; ++w)
            if (s.sw[w].col != STEPS || s.mom[w] != NBLK) return printf("violation deadlock\n"), 0;
        for (int p = 0; p < PR; ++p)
            if (s.out[p] != (1 << NBLK) - 1) return printf("violation block never written\n"), 0;
    }
    printf("ok %zu\n", seen.size());
}
