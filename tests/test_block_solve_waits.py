"""The block solve's waits that one lane makes for its warp: a failed one must not
send that lane on alone, or the others would wait for it in the next warp-wide
instruction (read from the source: a wait that runs out is not provoked on a
GPU)."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_2006_16117_gb300", "csrc", "solve_cluster.cu")


def _producers():
    s = open(SRC).read()
    return s[s.index("// ---- producers"): s.index("// ---- consumers")]


def test_no_lane_keeps_the_outcome_of_a_wait_for_itself():
    text = _producers()
    waits = [m.start() for m in re.finditer(r"\bbounded\(", text)]
    assert waits
    for at in waits:
        # up to the next warp-wide instruction; a wait that ran out has set s_fail
        nxt = re.search(r"__(shfl|syncwarp|any|all|ballot|reduce)\w*", text[at:])
        assert nxt is not None
        assert "break" not in text[at: at + nxt.start()] and "continue" not in text[at: at + nxt.start()]
        kept = re.search(r"(\w+) = $", text[:at])
        if kept:  # an outcome that is kept is handed to all lanes there
            args = text[at + nxt.end(): at + nxt.end() + 60]
            assert nxt.group(0).startswith("__shfl"), text[at: at + 200]
            assert re.match(r"\(0xffffffffu, \(int\)%s, 0\)" % kept.group(1), args), args
    # the check that ends the loop for the whole warp once s_fail is set
    assert re.search(r"if \(failed_flag\(&s_fail\)\) ok = false;\s*\}\s*ok = __shfl_sync\(0xffffffffu, \(int\)ok, 0\)", text)
    # and the copies in flight are waited for whichever lane or warp failed
    assert "if (pt == 0 && (!ok || failed_flag(&s_fail)))" in text


def test_recorded_wait_error_is_thrown_once(tmp_path):
    import native_program

    out = native_program.run(tmp_path, r'''
#include <cstdio>
#include "solve_cluster.h"
int main() {
    int code = 3, thrown = 0;
    sim::JobHost h;
    h.err = &code;
    for (int i = 0; i < 2; ++i) try {
        sim::block_solve_check(h);
    } catch (const sim::CudaError& e) {
        ++thrown;
        printf("%s\n", e.what.c_str());
    }
    h.err = nullptr;
    printf("%d %d\n", thrown, code);
}
''').splitlines()
    assert out[-1] == "1 0" and "code 3" in out[0], out


def test_inner_solve_reads_the_error_wherever_it_waits():
    s = open(os.path.join(os.path.dirname(SRC), "krylov.cu")).read()
    body = s[s.index("bool inner_solve(const Pencil& P"): s.index("// Arnoldi with CGS2 for all jobs")]
    waits = re.findall(r"cudaStreamSynchronize\(st\)\);\s*(\w+)", body)
    assert waits and set(waits) == {"block_solve_check"}, waits
