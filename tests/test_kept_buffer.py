"""A buffer that is kept clear between uses does not count as clear once it has
been allocated anew, also where the call that grew it fails afterwards
(csrc/lfd_kept.h, compiled for the host with an allocator of its own)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1812_06856_gb300", "csrc")

SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "lfd_kept.h"

static bool refuse = false;          // the next allocation fails

static int grow(void **p, size_t *cap, size_t bytes)
{
    if (*cap >= bytes) return 0;
    free(*p);
    *p = nullptr;
    *cap = 0;
    if (refuse) return 1;
    *p = malloc(bytes);
    memset(*p, 0x5a, bytes);         // not what the buffer is kept at
    *cap = bytes;
    return 0;
}

// a use as a fusion call makes it: 0 done, 1 refused; -1: it ran on words that are not clear
static int use(lfd::KeptBuffer<unsigned> &z, void **table, size_t *tcap, size_t bytes, bool fail_table)
{
    refuse = false;
    if (z.reserve(bytes, grow)) return 1;
    refuse = fail_table;
    if (grow(table, tcap, bytes)) return 1;
    if (!z.clean) memset(z.p, 0, z.cap);
    z.clean = false;
    for (size_t k = 0; k < z.cap / 4; k++)
        if (z.p[k]) return -1;
    z.clean = true;
    return 0;
}

int main()
{
    lfd::KeptBuffer<unsigned> z;
    void *table = nullptr;
    size_t tcap = 0;
    const int got[5] = {use(z, &table, &tcap, 64, false), use(z, &table, &tcap, 64, false), use(z, &table, &tcap, 4096, true),
                        use(z, &table, &tcap, 4096, false), use(z, &table, &tcap, 64, false)};
    printf("%d %d %d %d %d", got[0], got[1], got[2], got[3], got[4]);
    free(z.p);
    free(table);
    return 0;
}
"""


def test_a_failed_call_leaves_no_buffer_taken_for_clear(tmp_path):
    (tmp_path / "kept.cpp").write_text(SOURCE)
    exe = tmp_path / "kept"
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-I", CSRC, "-o", str(exe), str(tmp_path / "kept.cpp")])
    assert subprocess.run([str(exe)], capture_output=True, text=True).stdout == "0 0 1 0 0"
