"""The resident FP32 solve's dependencies, enumerated on the host from the functions that its kernel
waits and stores by (csrc/solve_order.h)."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2109_10277_gb300", "csrc")
SHIM = """
#include "solve_order.h"
extern "C" {
int node(int s, int n) { return hq::fold_node(s, n); }
int out_row(int p, int s, int n) { return hq::rs_out_row(p, s, n); }
int arrival(int p, int R, int blocks, int r, int b) { return hq::rs_arrival(p, R, blocks, r, b); }
int counters(int R, int blocks) { return hq::rs_counters(R, blocks); }
int wait(int p, int R, int blocks, int ntr, int r, int row0, int* target) {
  const hq::RsWait w = hq::rs_wait(p, R, blocks, ntr, r, row0);
  *target = w.target;
  return w.counter;
}
}
"""


@pytest.fixture(scope="module")
def order(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("order")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "shim.so")
    subprocess.run([gxx, "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "shim.cpp"), "-o", so], check=True)
    return C.CDLL(so)


@pytest.mark.parametrize("R", [1, 2, 5])
@pytest.mark.parametrize("bn", [32, 64])
@pytest.mark.parametrize("n", [256, 512])
def test_products_wait_for_every_producer(order, n, bn, R):
    """A product's tile may load its data rows once every tile of the product before that stores into
    them has reported: each such tile reports to the counter the wait reads, whose target is reached
    only by all the tiles that report to it.  Every counter lies within the kernel's range."""
    blocks, ntr = n // 128, n // bn
    assert sorted(order.node(s, n) for s in range(n)) == list(range(n))
    for p in (1, 2, 3):
        reports = {}   # counter -> tiles (right-hand side, slot block, data tile) of product p - 1
        writers = {}   # (right-hand side, row) -> slot block that stores it, for every data tile
        for r in range(R):
            for b in range(blocks):
                c = order.arrival(p - 1, R, blocks, r, b)
                assert 0 <= c < order.counters(R, blocks)
                reports.setdefault(c, set()).update((r, b, t) for t in range(ntr))
                for s in range(128 * b, 128 * (b + 1)):
                    writers[r, order.out_row(p - 1, s, n)] = b
        assert len(writers) == R * n
        for r in range(R):
            for row0 in range(0, n, bn):
                target = C.c_int()
                c = order.wait(p, R, blocks, ntr, r, row0, C.byref(target))
                assert target.value == len(reports[c])
                needed = {(r, writers[r, row], t) for row in range(row0, row0 + bn) for t in range(ntr)}
                assert needed <= reports[c], (p, row0)


@pytest.mark.parametrize("n", [256, 512])
def test_third_operand_may_be_overwritten(order, n):
    """Product 2 stores into the buffer that product 0 reads: its tiles start after every data tile of
    product 1 with one slot block, which together waited for all slot blocks of product 0."""
    blocks, ntr, bn = n // 128, n // 32, 32
    target = C.c_int()
    waited = {order.wait(1, 1, blocks, ntr, 0, t * bn, C.byref(target)) for t in range(ntr)}
    assert waited == {order.arrival(0, 1, blocks, 0, b) for b in range(blocks)}
