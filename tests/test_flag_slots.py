"""The borrowed (pinned word, event) slots of the graph set-up, with a fake source of both: host code only, built with g++."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_06354_b200", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <atomic>
#include "flag_slots.h"
static std::atomic<int> words{0}, events{0};
static bool refuse_event = false;
struct Fake {
    using Event = int;
    static bool make_word(int** w) { *w = new int(0); ++words; return true; }
    static void free_word(int* w) { delete w; --words; }
    static bool make_event(Event* e) { if (refuse_event) return false; *e = 1; ++events; return true; }
    static void free_event(Event) { --events; }
};
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
int main() {
    using Pool = gnn::FlagSlots<Fake>;
    const int kept = (int)gnn::FLAG_SLOTS_KEPT;
    Pool pool;
    Pool::Slot a, b;
    CHECK(pool.take(0, &a));
    int* const word = a.word;
    pool.give(a, true);
    CHECK(pool.take(1, &b) && b.word != word);  // another device's
    CHECK(pool.take(0, &a) && a.word == word);  // kept for the next call
    // a call whose kernels may still run does not hand its word to the next one
    pool.give(a, false);
    Pool::Slot c;
    CHECK(pool.take(0, &c) && c.word != word);
    pool.give(b, true);
    pool.give(c, true);
    // many calls at once leave a bounded number behind
    Pool::Slot many[40];
    const int before = words - 2;
    for (auto& s : many) CHECK(pool.take(0, &s));
    for (auto& s : many) pool.give(s, true);
    CHECK(words - before == kept && events - before == kept);
    refuse_event = true;
    CHECK(!pool.take(7, &a) && words - before == kept);  // no event: the word goes back
    refuse_event = false;
    // no word in two hands
    std::atomic<int> clashes{0};
    std::thread t[8];
    for (auto& th : t) th = std::thread([&] {
        for (int i = 0; i < 20000; ++i) {
            Pool::Slot s;
            if (!pool.take(0, &s)) { ++clashes; return; }
            if (__atomic_fetch_add(s.word, 1, __ATOMIC_RELAXED) != 0) ++clashes;
            __atomic_fetch_sub(s.word, 1, __ATOMIC_RELAXED);
            pool.give(s, true);
        }
    });
    for (auto& th : t) th.join();
    CHECK(clashes == 0 && words - before <= kept);
    return 0;
}
"""


def test_slots_are_bounded_and_never_shared(tmp_path):
    src, exe = tmp_path / "slots.cpp", tmp_path / "slots"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I" + CSRC, str(src), "-o", str(exe)], check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
