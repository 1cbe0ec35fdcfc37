"""Host-side bookkeeping of the library, compiled from its headers with the host compiler (no GPU needed)."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_20564_b200", "csrc")


def run_cpp(tmp_path, body, *headers):
    """Compiles and runs `body` as main(); it returns 0 when all is well, else the number of the check that failed."""
    src = tmp_path / "t.cpp"
    src.write_text("".join(f'#include "{h}"\n' for h in headers) + "#include <string>\nusing namespace e2egrec;\n"
                   "int main() {\n" + body + "\nreturn 0;\n}\n")
    exe = tmp_path / "t"
    subprocess.check_call(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)])
    assert subprocess.call([str(exe)], timeout=60) == 0


LEDGER = """
DeferralLedger led;
std::string log;
uint64_t capture = 0;
auto join = [&](size_t who) {
    log.clear();
    led.join(who, [&] { return capture; }, [&](size_t h) { log += char('A' + h); });
    return log;
};
enum : size_t { A, B, C };
"""


def test_every_stream_waits_once_for_every_deferral(tmp_path):
    run_cpp(tmp_path, LEDGER + """
if (join(A) != "") return 1;
led.defer(A, 0);
if (join(B) != "A") return 2;          // an unrelated stream asks first ...
if (join(A) != "A") return 3;          // ... and the owner, about to use the scratch again, still waits
if (join(A) != "" || join(B) != "") return 4;
if (join(C) != "A") return 5;
led.defer(A, 0);                       // two callers, each with its own sample
led.defer(B, 0);
if (join(A) != "AB" || join(B) != "AB" || join(A) != "") return 6;
led.defer(A, 0);
led.defer(A, 0);
if (join(A) != "A" || join(A) != "") return 7;
""", "deferral.h")


def test_waits_and_stream_captures(tmp_path):
    run_cpp(tmp_path, LEDGER + """
capture = 7;                           // deferred and joined inside one capture, by two of its streams
led.defer(A, 7);
if (join(B) != "A" || join(A) != "A") return 1;
led.defer(A, 7);
if (join(B) != "A") return 2;
capture = 0;                           // the capture has ended: its events are no longer to be waited for
if (join(A) != "") return 3;
led.defer(A, 0);
if (join(B) != "A") return 4;
capture = 8;                           // no wait for outside work inside a capture, unless nobody has waited for it
if (join(A) != "") return 5;
capture = 0;                           // the owner's next call outside makes up for it
if (join(A) != "A" || join(A) != "") return 6;
led.defer(A, 0);
capture = 9;
if (join(A) != "A") return 7;          // refused by CUDA, as a join of another capture's work always was
""", "deferral.h")


def test_walks_end_with_offsets_that_decrease(tmp_path):
    """A search that keeps returning the same segment, or one further back, does not hold the walk; one that finds a segment
    ahead is followed; numbers beyond 2^31 are fine."""
    run_cpp(tmp_path, """
const int64_t n = 1000;
for (int64_t stuck : {int64_t(0), int64_t(40), n - 1}) {
    int64_t base = 5;
    for (int windows = 0; base < n; ++windows) {
        if (windows > n / 32 + 1) return 1;
        base = window_found(base, stuck);
    }
}
if (window_found(int64_t(64), int64_t(500)) != 500) return 2;
if (window_found(uint32_t(2147483647u), 0u) != 2147483679u) return 3;
""", "stdint.h", "window.h")


def test_rows_of_entries_behind_the_last_offset(tmp_path):
    """The row expansion's walk over 32 rows at a time, for offsets that end with the entries and for offsets that end before
    them, with the last rows empty or not: every entry's row, and never one beyond the last."""
    run_cpp(tmp_path, """
for (int n_rows : {1, 31, 32, 33, 64, 100})
    for (int tail : {0, 1, 40})                              // empty rows at the end
        for (int extra : {0, 5, 200}) {                      // entries that the offsets do not cover
            std::vector<int64_t> ptr(1, 0);
            for (int r = 0; r < n_rows; ++r) ptr.push_back(ptr.back() + (r < n_rows - tail ? r % 4 : 0));
            const int m = (int)ptr.back() + extra;
            for (int k0 = 0; k0 < m; k0 += 48) {             // spans
                const int len = std::min(48, m - k0);
                int64_t base = 0;
                while (base + 1 < n_rows && ptr[base + 1] <= k0) ++base;
                std::vector<int32_t> row(len, -1);
                row[0] = (int32_t)base;
                auto begin = [&](int64_t r) { return r <= n_rows ? (int)std::max<int64_t>(std::min<int64_t>(ptr[r] - k0, 48), 0) : 48; };
                for (;; base += 32) {
                    for (int lane = 0; lane < 32; ++lane) {
                        const int beg = begin(base + lane);
                        const int32_t noted = row_to_note(base + lane, n_rows, beg, begin(base + lane + 1), len);
                        if (noted >= 0) row[beg] = noted;
                    }
                    if (!more_rows(base, n_rows, begin(base + 32), len)) break;
                }
                for (int e = 0; e < len; ++e) {
                    if (e && row[e] < 0) row[e] = row[e - 1];
                    int64_t want = 0;
                    while (want + 1 < n_rows && ptr[want + 1] <= k0 + e) ++want;
                    if (row[e] != want) return 1;
                }
            }
        }
""", "algorithm", "vector", "window.h")
