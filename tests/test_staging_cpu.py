"""Host descriptor blocks of asynchronous copies (staging.h) under the latest copies that the CUDA runtime
allows: a source is read only when the stream is waited for.  Every copy has to find the bytes that were
in its block when it was issued, also with more copies than blocks, and the ring waits when it goes away
early.  Host code only."""
import ctypes
import os
import subprocess

import pytest

from paper_2406_14084_gb300 import qs

CODE = r"""
#include <cstring>
#include <utility>
#include "staging.h"
extern "C" int late_copies(int copies, int blocks, int leave, int *waits)
{
    std::vector<std::pair<int, const int *>> queue;  // expected value, source
    int seen = 0, wrong = 0;
    *waits = 0;
    auto wait = [&] {
        ++*waits;
        for (auto &c : queue) {
            for (int i = 0; i < 8; ++i) wrong += c.second[i] != c.first;
            ++seen;
        }
        queue.clear();
    };
    {
        qs::StagingRing<decltype(wait)> ring(8 * sizeof(int), blocks, wait);
        for (int k = 0; k < copies; ++k) {
            int *p = static_cast<int *>(ring.next());
            for (int i = 0; i < 8; ++i) p[i] = k;
            queue.push_back({k, p});
        }
        if (!leave) {  // the caller's own synchronize
            wait();
            ring.idle();
        }
    }
    return wrong + (seen != copies);
}
"""


@pytest.fixture(scope="module")
def late_copies(tmp_path_factory):
    d = tmp_path_factory.mktemp("staging")
    src, so = d / "late.cpp", d / "late.so"
    src.write_text(CODE)
    csrc = os.path.join(os.path.dirname(os.path.abspath(qs.__file__)), "csrc")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", csrc, str(src), "-o", str(so)], check=True)
    return ctypes.CDLL(str(so)).late_copies


@pytest.mark.parametrize("leave", [0, 1])
@pytest.mark.parametrize("copies", [0, 1, 4, 5, 13])
def test_every_copy_finds_its_bytes(late_copies, copies, leave):
    waits = ctypes.c_int()
    assert late_copies(copies, 4, leave, ctypes.byref(waits)) == 0
    full = max(0, (copies - 1) // 4)  # one wait each time a block is wanted and all are in use
    assert waits.value == full + (1 if not leave or copies else 0)
