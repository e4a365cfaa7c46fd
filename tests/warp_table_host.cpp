// Runs csrc/warp_table.cuh on the host: the 32 lanes are coroutines, switched
// in random order before every access to the table, so that only the warp
// barriers order them.  Prints the first violated property and returns 1.
#include <stdio.h>
#include <stdlib.h>
#include <ucontext.h>

#include <random>
#include <set>
#include <utility>
#include <vector>

constexpr int LANES = 32;
static ucontext_t main_cx, lane_cx[LANES];
static std::vector<char> stack_of[LANES];
static int cur;
static enum { RUN, WAIT, DONE } state[LANES];
static bool pred[LANES], vote;

static void yield() { swapcontext(&lane_cx[cur], &main_cx); }
static void barrier()
{
    state[cur] = WAIT;
    yield();
}
static void __syncwarp() { barrier(); }
static int __any_sync(unsigned, bool p)
{
    pred[cur] = p;
    barrier();
    return vote;
}
#define __device__
#define __forceinline__ inline
#include "../paper_2006_14956_gb300/csrc/warp_table.cuh"

struct Slot {
    int *p;
    operator int() const { yield(); return *p; }
    void operator=(int v) const { yield(); *p = v; }
};
struct Table {
    int *t;
    Slot operator[](unsigned s) const { return Slot{t + s}; }
};

static std::mt19937 rng;
static void (*body)(int);
static void entry(int lane)
{
    body(lane);
    state[lane] = DONE;
    swapcontext(&lane_cx[lane], &main_cx);
}
static void run_warp(void (*f)(int))
{
    body = f;
    for (int l = 0; l < LANES; l++) {
        stack_of[l].resize(1 << 16);
        getcontext(&lane_cx[l]);
        lane_cx[l].uc_stack.ss_sp = stack_of[l].data();
        lane_cx[l].uc_stack.ss_size = stack_of[l].size();
        lane_cx[l].uc_link = &main_cx;
        state[l] = RUN;
        makecontext(&lane_cx[l], (void (*)())entry, 1, l);
    }
    for (;;) {
        int ready[LANES], n = 0, waiting = 0;
        for (int l = 0; l < LANES; l++) {
            if (state[l] == RUN) ready[n++] = l;
            waiting += state[l] == WAIT;
        }
        if (!n) {
            if (!waiting) return;
            vote = false;
            for (int l = 0; l < LANES; l++) {
                vote |= state[l] == WAIT && pred[l];
                if (state[l] == WAIT) state[l] = RUN;
            }
            continue;
        }
        cur = ready[rng() % n];
        swapcontext(&main_cx, &lane_cx[cur]);
    }
}

constexpr int SLOTS = 128, ROUNDS = 3, NONE = 255;
static int tab[SLOTS], key[ROUNDS * LANES], start_slot[64], target[ROUNDS * LANES], round0;
static bool on[ROUNDS * LANES], distinct;
static void lane_body(int lane)
{
    const int e = round0 + lane, k = key[e];
    target[e] = fq::warp_claim(Table{tab}, (unsigned)SLOTS - 1, (unsigned)start_slot[k], e, (int)NONE, on[e],
                               [&](int x) { return !distinct && key[x] == k; });
}

int main(int argc, char **argv)
{
    const int trials = argc > 1 ? atoi(argv[1]) : 2000;
    for (int trial = 0; trial < trials; trial++) {
        rng.seed(trial);
        // few keys on few start slots: equal keys and collisions in every turn;
        // every fourth trial all keys distinct and never compared (walkers, list index)
        distinct = trial % 4 == 3;
        const int keys = 2 + (int)(rng() % 12), starts = 1 + (int)(rng() % 4);
        for (int k = 0; k < 64; k++) start_slot[k] = (int)(rng() % starts) * 3;
        for (int s = 0; s < SLOTS; s++) tab[s] = NONE;
        std::set<std::pair<int, int>> pairs;
        for (int r = 0; r < (distinct ? 1 : ROUNDS); r++) {
            round0 = r * LANES;
            for (int l = 0; l < LANES; l++) {
                key[round0 + l] = distinct ? l : (int)(rng() % keys);
                on[round0 + l] = rng() % 8 != 0;
            }
            run_warp(lane_body);
            for (int l = 0; l < LANES; l++) {
                const int e = round0 + l, t = target[e];
                if (!on[e]) {
                    if (t != -1) { printf("trial %d: an idle lane found a record\n", trial); return 1; }
                    continue;
                }
                if (t < 0 || key[t] != key[e] || target[t] != t) {
                    printf("trial %d: record %d points to %d\n", trial, e, t);
                    return 1;
                }
                pairs.insert({key[e], t});
            }
            std::set<int> owners, in_table;
            for (auto &p : pairs) owners.insert(p.first);
            if (owners.size() != pairs.size()) { printf("trial %d: a key has two records\n", trial); return 1; }
            int used = 0;
            for (int s = 0; s < SLOTS; s++)
                if (tab[s] != NONE) { used++; in_table.insert(tab[s]); }
            if (used != (int)pairs.size() || in_table.size() != pairs.size()) {
                printf("trial %d: %d slots for %d records\n", trial, used, (int)pairs.size());
                return 1;
            }
        }
    }
    return 0;
}
