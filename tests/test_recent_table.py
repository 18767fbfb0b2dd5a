"""The table of what a thread has worked out before (csrc/recent.h), compiled on its own: layers in rotation are worked out once,
and what is in use does not give way to what is not."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_14811_b200", "csrc")
PROGRAM = r"""
#include <cstdio>
#include "recent.h"
struct Key { int64_t M, N, K; bool operator==(const Key &o) const { return M == o.M && N == o.N && K == o.K; } };
static int worked_out = 0;
static sq::Recent<Key, int64_t, 8, 32> kept;
static uint32_t hash_of(const Key &k) { const int64_t w[3] = {k.M, k.N, k.K}; return sq::hash_words(w, 3); }
static bool ask(const Key &k)                                     // true: the value is the key's own
{
    const uint32_t h = hash_of(k);
    if (const int64_t *v = kept.find(h, k)) return *v == k.M * k.N + k.K;
    worked_out++;
    return kept.keep(h, k, k.M * k.N + k.K) == k.M * k.N + k.K;
}
int main()
{
    bool ok = true;
    for (int round = 0; round < 50; round++)                      // a text stream of 20 lengths through 8 layer shapes
        for (int M = 77; M < 97; M++)
            for (int s = 0; s < 8; s++) ok &= ask({M, 1152 * (1 + s % 4), 768 << s / 4});
    std::printf("%d ", worked_out);
    const Key hot{8, 18432, 3072};
    worked_out = 0;
    int hot_again = 0;
    ok &= ask(hot);
    for (int M = 1; M <= 20000; M++) {                            // ever new shapes, one layer in use among them
        ok &= ask({M, 640, 1280});
        const int before = worked_out;
        ok &= ask(hot);
        hot_again += worked_out - before;
    }
    std::printf("%d %d\n", hot_again, int(ok));
}
"""


def test_layers_in_rotation_are_worked_out_once(tmp_path):
    source, program = tmp_path / "recent.cpp", tmp_path / "recent"
    source.write_text(PROGRAM)
    subprocess.check_call([os.environ.get("CXX", "g++"), "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC, str(source), "-o", str(program)])
    once, hot_again, ok = map(int, subprocess.check_output([str(program)]).split())
    assert (once, hot_again, ok) == (160, 0, 1)
