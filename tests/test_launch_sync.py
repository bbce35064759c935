"""What a launch may rely on when it looks the tree up before it waits for its
predecessor (TreeSync), as the host hands it out: nothing older than the last
remesh, and no count that an earlier launch could have left."""
import subprocess

SRC = r"""
#include <cstdio>
#include "mrlt_tree.cuh"
using namespace mrlt;
int main(int argc, char** argv)
{
    Launcher K;
    for (const char* c = argv[1]; *c; ++c) {
        if (*c == '[') { K.capturing = true; K.stale = false; K.published[0] = 0; K.stages = 0; } // piece_begin
        else if (*c == ']') { K.capturing = false; K.stale = true; }                             // piece_end
        else if (*c == 'w') K.wait_first = true;
        else if (*c == 'c') K.stale = true; // compaction, resize, fine step, graph launch
        else {
            const TreeSync s = K.enter();
            printf("%d %d %u\n", s.mode, s.word, s.need);
        }
    }
    return 0;
}
"""
VISIBLE, ACQUIRE, PUBLISH, WAIT = range(4)


def test_entry_of_launches(tmp_path):
    from paper_1905_08717_gb300 import build as b
    (tmp_path / "t.cu").write_text(SRC)
    exe = str(tmp_path / "t")
    subprocess.check_call([b._nvcc()] + b.ARCH + ["-std=c++17", "-I" + b.CSRC, "-o", exe, str(tmp_path / "t.cu")])

    def run(seq):
        return [tuple(map(int, r.split())) for r in subprocess.check_output([exe, seq], text=True).splitlines()]

    # captured: everything before the piece is visible; after each remesh one
    # launch waits and publishes, and the others need its count
    assert run("[eecececc" "ee]") == [(VISIBLE, 0, 0), (VISIBLE, 0, 0), (PUBLISH, 0, 1), (PUBLISH, 0, 2),
                                      (PUBLISH, 0, 3), (ACQUIRE, 0, 3)]
    assert run("[cee][eec" "e]") == [(PUBLISH, 0, 1), (ACQUIRE, 0, 1), (VISIBLE, 0, 0), (VISIBLE, 0, 0), (PUBLISH, 0, 1)]
    # direct: the first launch waits and publishes; the count only grows, also
    # over captured pieces between
    assert run("eecee") == [(PUBLISH, 1, 1), (ACQUIRE, 1, 1), (PUBLISH, 1, 2), (ACQUIRE, 1, 2)]
    got = run("ee[ecee]eece")
    assert got == [(PUBLISH, 1, 1), (ACQUIRE, 1, 1), (VISIBLE, 0, 0), (PUBLISH, 0, 1), (ACQUIRE, 0, 1),
                   (PUBLISH, 1, 2), (ACQUIRE, 1, 2), (PUBLISH, 1, 3)]
    # a solver that waits first does so everywhere
    assert {m for m, _, _ in run("we[eece]ece")} == {WAIT}
