"""Initial data at any address.  Large data may be read in place by a kernel,
which loads whole doubles: only arrays on their boundary may take that way, all
others are copied.  The rule is tested on the host, every combination; the
calls on the GPU, with arrays behind an odd offset on either side of the size
from which data are read in place."""
import os
import subprocess

import numpy as np
import pytest

from paper_1905_08717_gb300 import inputs as I

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdio>
#include <initializer_list>
#include "mrlt_input.h"
int main()
{
    for (int offset = 0; offset < 16; ++offset)
        for (size_t bytes : {mrlt::kReadInPlace - 8, mrlt::kReadInPlace, mrlt::kReadInPlace + 8})
            for (int lived = 0; lived < 2; ++lived)
                for (int tables = 0; tables < 2; ++tables)
                    printf("%d %lld %d %d %d\n", offset, (long long)bytes - (long long)mrlt::kReadInPlace, lived, tables,
                           (int)mrlt::read_in_place((const void*)(uintptr_t)(4096 + offset), bytes, lived, tables));
    return 0;
}
"""


def test_rule(tmp_path):
    (tmp_path / "t.cpp").write_text(SRC)
    exe = str(tmp_path / "t")
    subprocess.check_call(["g++", "-std=c++17", "-I" + os.path.join(ROOT, "paper_1905_08717_gb300", "csrc"), "-o", exe,
                           str(tmp_path / "t.cpp")])
    rows = [tuple(map(int, r.split())) for r in subprocess.check_output([exe], text=True).splitlines()]
    assert len(rows) == 16 * 3 * 2 * 2
    for offset, over, lived, tables, placed in rows:
        assert placed == (offset % 8 == 0 and over >= 0 and not lived and bool(tables)), (offset, over, lived, tables)


def _at_offset(q, offset):
    """q in an array whose first byte lies `offset` bytes behind an 8-byte boundary"""
    buf = bytearray(q.nbytes + 32)
    start = (-np.frombuffer(buf, np.uint8).ctypes.data) % 8 + offset
    out = np.frombuffer(buf, np.float64, q.size, start).reshape(q.shape)
    out[...] = q
    assert out.ctypes.data % 8 == offset
    return out


@pytest.mark.gpu
@pytest.mark.parametrize("L", [8, 10])  # 2.1 MB, 33.5 MB
def test_unaligned_arrays(L):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1905_08717_gb300 as pkg
    from paper_1905_08717_gb300 import build
    build.build()
    p, q = I.euler_2d_quadrants(L=L, seed=3)
    q2 = np.ascontiguousarray(I.euler_2d_quadrants(L=L, seed=4)[1])

    def results(f):
        s = pkg.Solver(p, f(q))
        s.step(0.002)
        out = list(s.leaves())
        s.reset(f(q2))
        out += s.leaves()
        s.close()
        b = pkg.Batch([p], [f(q2)])
        out += b.instances[0].leaves()
        b.close()
        v = pkg.Server(8 << 30, 2)
        rid = v.submit(p, f(q), 0.002)
        while not v.poll():
            v.advance()
        out += v.result(rid).leaves()
        v.close()
        return out

    want = results(lambda a: np.ascontiguousarray(a))
    for offset in (1, 4):
        for a, b in zip(want, results(lambda x: _at_offset(np.ascontiguousarray(x), offset))):
            assert np.array_equal(a, b), offset
