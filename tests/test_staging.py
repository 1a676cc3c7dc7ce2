"""The ring of slots of csrc/lbm_staging.h with a fake device, on the host: every
chunk arrives, a slot is never reused before its last use has ended, and after a
failed launch or wait nothing is outstanding when the call returns."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_20650_gb300", "csrc")

SOURCE = r"""
#include "lbm_staging.h"
#include <cstdio>
#include <cstdlib>
#include <mutex>
#include <vector>

// The fake device does a launch's work when it is awaited, or at the next launch
// after two more (late), so a slot touched in between shows.
struct Fake {
    int64_t chunks;
    bool to_host;
    int64_t bad_launch, bad_wait;
    std::vector<int64_t> array;
    int64_t slot[lbm::kStageSlots], pending[lbm::kStageSlots];
    std::atomic<int> copying{0};
    std::atomic<bool> wrong{false};
    int64_t waits = 0;
    Fake(int64_t n, bool h, int64_t bl, int64_t bw) : chunks(n), to_host(h), bad_launch(bl), bad_wait(bw), array(n, -1) {
        for (auto &p : pending) p = -1;
        for (auto &s : slot) s = -1;
        if (!h) for (int64_t c = 0; c < n; ++c) array[c] = 7 * c + 1;
    }
    std::vector<int64_t> device = std::vector<int64_t>(chunks, -1);
    bool launch(int64_t c, int s) {
        if (c == bad_launch) return false;
        if (pending[s] != -1) wrong = true;            // still in use by the device
        if (to_host && slot[s] != -1) wrong = true;    // not yet emptied by the host
        pending[s] = c;
        return true;
    }
    bool wait(int s) {
        const int64_t c = pending[s];
        if (c == -1) wrong = true;
        else if (to_host) slot[s] = 7 * c + 1;
        else { device[c] = slot[s]; slot[s] = -1; }
        pending[s] = -1;
        return waits++ != bad_wait;
    }
    void copy(int64_t c, int s) {
        copying++;
        if (to_host) { array[c] = slot[s]; slot[s] = -1; }
        else {
            if (slot[s] != -1) wrong = true;           // the device has not read the last chunk
            slot[s] = array[c];
        }
        if (c % 3 == 0) std::this_thread::yield();
        copying--;
    }
};

int main() {
    const int64_t sizes[] = {0, 1, 2, 3, 15, 16, 17, 33, 200};
    for (int64_t n : sizes)
        for (int workers : {0, 1, 3, 15})
            for (int h = 0; h < 2; ++h)
                for (int64_t bad = -1; bad < n; bad += bad < 3 ? 1 : 13)
                    for (int kind = 0; kind < 2; ++kind) {
                        Fake io(n, h, kind == 0 ? bad : -1, kind == 1 ? bad : -1);
                        const bool ok = lbm::staged_transfer(io, n, workers, h != 0);
                        bool good = !io.wrong && io.copying == 0 && ok == (bad < 0);
                        for (int64_t p : io.pending) good = good && p == -1;
                        for (int64_t c = 0; c < n && bad < 0; ++c)
                            good = good && (h ? io.array[c] : io.device[c]) == 7 * c + 1;
                        if (!good) {
                            printf("n %ld workers %d to_host %d bad %ld kind %d\n", (long)n, workers, h, (long)bad, kind);
                            return 1;
                        }
                    }
    return 0;
}
"""


@pytest.mark.parametrize("flags", [["-O2"], ["-O1", "-g", "-fsanitize=thread"]], ids=["plain", "thread checker"])
def test_ring_of_slots(tmp_path, flags):
    src, exe = tmp_path / "staging.cpp", tmp_path / "staging"
    src.write_text(SOURCE)
    r = subprocess.run(["g++", "-std=c++17", *flags, "-I", CSRC, str(src), "-o", str(exe), "-pthread"],
                       capture_output=True, text=True)
    if r.returncode != 0 and "thread" in " ".join(flags):
        pytest.skip("no thread checker: " + r.stderr[-200:])
    assert r.returncode == 0, r.stderr
    for _ in range(3):
        r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
        if "unexpected memory mapping" in r.stderr:
            pytest.skip("the thread checker does not run on this kernel")
        assert r.returncode == 0, r.stdout + r.stderr
