"""How the two softmax warps that share a row keep one reference, as a model on the host over the kernel's own rule: every order
in which scores land, words are posted and read, and P is handed over.  From every state the end can be reached, and every order
ends with the same references and the same roundings."""
import os
import subprocess

from paper_2602_15318_b200 import build

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_15318_b200", "csrc")

MODEL = r"""
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <map>
#include <string>
#include <vector>
#include "softmax_pair.cuh"
using namespace sparrow::tc;

// The kernel's order, and mistakes: P handed over and the next tile looked at whether or not the partner has passed this one; a
// move posted over one that the partner has not read; a move held back until the partner has passed the same tile.
struct Kernel {
    static bool may_settle(int j, int word) { return pair_passed(word) > j; }
    static bool may_post(int j, int word) { return pair_settled(word, j - 1); }
};
struct Unbound : Kernel { static bool may_settle(int, int) { return true; } };
struct Overwrites : Kernel { static bool may_post(int, int) { return true; } };
struct WaitsForPass : Kernel { static bool may_post(int j, int word) { return pair_passed(word) > j; } };

constexpr int kMost = 7, kBlocks = 3;         // tiles; score blocks
enum { POLL, SETTLE, LOOK, POST, HAND, WORK, FIRST, LAST, DONE };
struct Warp { signed char pc, j, handed, ref, acc, moved, cand; };
struct State {
    Warp w[2];
    signed char word[2], posted[2], landed, pad;
    signed char p_ref[2][kMost][4];           // references that a tile's P has gone through
    signed char o_ref[2][kMost];              // reference of each half of O in front of a tile's product
};
struct Result { long states, stuck, ends, wrong; };

// score[w][t]: the largest score of warp w's half of tile t (-1: all masked); a reference moves where it is exceeded
template <class Rule>
Result explore(int n, const signed char (&score)[2][kMost])
{
    State s0;
    std::memset(&s0, 0, sizeof s0);
    for (Warp& w : s0.w) { w.pc = POLL; w.ref = w.acc = -1; }
    std::map<std::string, int> seen;
    std::vector<State> all;
    std::vector<std::vector<int>> from;
    Result r = {0, 0, 0, 0};
    auto add = [&](const State& s, int parent) {
        const std::string key(reinterpret_cast<const char*>(&s), sizeof s);
        auto it = seen.find(key);
        if (it == seen.end()) { it = seen.emplace(key, (int)all.size()).first; all.push_back(s); from.emplace_back(); }
        if (parent >= 0) from[it->second].push_back(parent);
    };
    add(s0, -1);
    for (size_t at = 0; at < all.size(); ++at) {
        const State s = all[at];
        // the next tile's scores land: at once where there is a block for them, else behind the product that frees it
        if (s.landed < n && (s.landed < kBlocks || std::min(s.w[0].handed, s.w[1].handed) > s.landed - kBlocks)) {
            State x = s;
            ++x.landed;
            add(x, (int)at);
        }
        for (int i = 0; i < 2; ++i) {
            State x = s;
            Warp& w = x.w[i];
            const int partner = x.word[i ^ 1], j = w.j;
            switch (w.pc) {
            case POLL:                         // (at the end there is no tile to wait for)
                if (j < n && j >= x.landed) continue;
                w.pc = j > 0 ? SETTLE : LOOK;
                break;
            case SETTLE: {                     // the tile before
                const int t = j - 1;
                if (!Rule::may_settle(t, partner)) continue;
                const bool other = pair_passed(partner) > t && pair_moved(partner, t);
                if (pair_passed(partner) > t + 2) ++r.wrong;
                if (!pair_quiet(partner, t) || w.moved) {
                    signed char ref = w.ref;
                    if (other) ref = std::max(ref, x.posted[i ^ 1]);
                    if (ref != w.ref) x.p_ref[i][t][1] = ref + 2;
                    w.ref = w.acc = ref;
                    if (other) x.word[i] = pair_word(j, true, w.moved);
                }
                x.o_ref[i][t] = w.acc + 2;
                w.pc = j < n ? LOOK : HAND;
                break;
            }
            case LOOK: {
                const bool moves = score[i][j] > w.ref;
                w.moved = (w.moved << 1) & 3;
                if (j == 0) { x.posted[i] = w.cand = score[i][0]; w.pc = FIRST; break; }
                if (moves) { w.moved |= 1; w.cand = score[i][j]; w.pc = POST; }
                else { x.word[i] = pair_word(j + 1, false, w.moved); w.pc = HAND; }
                break;
            }
            case POST:                         // (looked at again and again)
                if ((w.moved & 2) && !Rule::may_post(j, partner)) continue;
                x.posted[i] = w.cand;
                w.ref = w.cand;
                x.word[i] = pair_word(j + 1, false, w.moved);
                w.pc = HAND;
                break;
            case HAND:                         // P of the tile before
                ++w.handed;
                w.pc = j < n ? WORK : LAST;
                break;
            case WORK:
                x.p_ref[i][j][0] = w.ref + 2;
                ++w.j;
                w.pc = POLL;
                break;
            case FIRST:
                if (i == 1 || x.w[1].pc != FIRST) continue;
                for (int v = 0; v < 2; ++v) {
                    x.w[v].ref = x.w[v].acc = std::max(x.posted[0], x.posted[1]);
                    x.word[v] = pair_word(1, false, 0);
                    x.w[v].pc = WORK;
                }
                break;
            case LAST:
                if (i == 1 || x.w[1].pc != LAST) continue;
                x.w[0].pc = x.w[1].pc = DONE;
                if (x.w[0].ref != x.w[1].ref) ++r.wrong;
                for (int t = 0; t < n; ++t) {                   // one reference for both halves of a tile, P and accumulator
                    signed char last[2];
                    for (int v = 0; v < 2; ++v) last[v] = x.p_ref[v][t][1] ? x.p_ref[v][t][1] : x.p_ref[v][t][0];
                    if (last[0] != last[1] || x.o_ref[0][t] != last[0] || x.o_ref[1][t] != last[0]) ++r.wrong;
                }
                break;
            default: continue;
            }
            add(x, (int)at);
        }
    }
    std::vector<char> good(all.size(), 0);
    std::vector<int> todo;
    for (size_t k = 0; k < all.size(); ++k)
        if (all[k].w[0].pc == DONE && all[k].w[1].pc == DONE) { good[k] = 1; ++r.ends; todo.push_back((int)k); }
    while (!todo.empty()) {
        const int k = todo.back();
        todo.pop_back();
        for (int p : from[k]) if (!good[p]) { good[p] = 1; todo.push_back(p); }
    }
    r.states = (long)all.size();
    r.stuck = (long)std::count(good.begin(), good.end(), 0);
    return r;
}

struct Sums { long cases, stuck, several, wrong; };
template <class Rule>
Sums over_all(int most, int step)
{
    Sums s = {0, 0, 0, 0};
    for (int n = 1; n <= most; ++n)
        for (int a = 0; a < 2 * n; ++a)                       // up to four places where scores grow, or are masked
            for (int b = a; b < 2 * n; ++b)
                for (int c = b; c < 2 * n; c += step)
                    for (int d = c; d < 2 * n; d += step)
                        for (int kind = 0; kind < 16; ++kind) {
                            signed char score[2][kMost] = {};
                            score[a % 2][a / 2] = kind & 1 ? 2 : -1;
                            score[b % 2][b / 2] = kind & 2 ? 3 : 1;
                            score[c % 2][c / 2] = kind & 4 ? 2 : 4;
                            score[d % 2][d / 2] = kind & 8 ? 5 : 3;
                            const Result r = explore<Rule>(n, score);
                            ++s.cases;
                            s.stuck += r.stuck > 0;
                            s.several += r.ends > 1;
                            s.wrong += r.wrong > 0;
                        }
    return s;
}

int main()
{
    const Sums k = over_all<Kernel>(6, 1), mistakes[3] = {over_all<Unbound>(4, 2), over_all<Overwrites>(4, 2), over_all<WaitsForPass>(3, 1)};
    std::printf("%d %ld %ld %ld %d %d %d\n", k.cases > 20000, k.stuck, k.several, k.wrong,
                mistakes[0].several + mistakes[0].wrong > 0, mistakes[1].several > 0, mistakes[2].stuck > 0);
    std::fprintf(stderr, "%ld cases; mistakes (stuck, several ends, wrong):", k.cases);
    for (const Sums& m : mistakes) std::fprintf(stderr, " %ld %ld %ld of %ld;", m.stuck, m.several, m.wrong, m.cases);
    return 0;
}
"""


def test_no_order_of_events_leaves_a_pair_waiting_or_changes_its_results(tmp_path):
    src, exe = tmp_path / "pair.cu", tmp_path / "pair"
    src.write_text(MODEL)
    subprocess.run([build.nvcc(), *build.NVCC_FLAGS[:2], "-O2", "-std=c++17", "-I" + CSRC, "-o", str(exe), str(src)], check=True, timeout=600)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=600)
    cases, stuck, several, wrong, *mistakes = r.stdout.split()
    assert r.returncode == 0 and cases == "1"
    assert stuck == "0", r.stderr                       # every state leads to the end
    assert several == "0", r.stderr                     # one end, whatever the order: references, roundings
    assert wrong == "0", r.stderr                       # both halves of P and of the accumulator on one reference at every product
    assert mistakes == ["1", "1", "1"], r.stderr        # the model shows what each mistake leads to
