"""Writes sort16_network.inc: Batcher's odd-even merge sort for 16 inputs as a list of
compare-exchange steps TDQ_CE(i, j) (i < j; the smaller value ends in slot i).

The eight steps on neighbours (2 i, 2 i + 1) come first, with the line TDQ_PAIRS behind them: the larger of each pair then
stands in the odd slots, and the includer takes the maximum of all sixteen from there (no step before them touches a slot
of theirs, so the order changes nothing).

The network is checked here with the 0-1 principle (all 65536 binary inputs) before it
is written.  The CUDA quantizer includes the file twice-unrolled in registers and uses
only the lowest few outputs, so the compiler drops the comparators that cannot reach them.

Run:  python gen_sort16.py
"""
import os


def batcher(n):
    steps = []

    def merge(lo, hi, r):
        step = 2 * r
        if step < hi - lo:
            merge(lo, hi, step)
            merge(lo + r, hi, step)
            for i in range(lo + r, hi - r, step):
                steps.append((i, i + r))
        else:
            steps.append((lo, lo + r))

    def sort(lo, hi):
        if hi > lo:
            mid = lo + (hi - lo) // 2
            sort(lo, mid)
            sort(mid + 1, hi)
            merge(lo, hi, 1)

    sort(0, n - 1)
    pairs = [(i, i + 1) for i in range(0, n, 2)]
    return pairs + [s for s in steps if s not in pairs]


def sorts_all_binary_inputs(steps, n):
    for bits in range(1 << n):
        v = [(bits >> i) & 1 for i in range(n)]
        for a, b in steps:
            if v[a] > v[b]:
                v[a], v[b] = v[b], v[a]
        if any(v[i] > v[i + 1] for i in range(n - 1)):
            return False
    return True


if __name__ == "__main__":
    net = batcher(16)
    assert len(net) == 63 and sorts_all_binary_inputs(net, 16)
    path = os.path.join(os.path.dirname(os.path.abspath(__file__)), "sort16_network.inc")
    with open(path, "w") as f:
        f.write("// Generated by gen_sort16.py: Batcher odd-even merge sort, 16 inputs, 63 steps.\n")
        for n, (a, b) in enumerate(net):
            f.write("TDQ_CE(%d, %d)\n" % (a, b) + ("TDQ_PAIRS\n" if n == 7 else ""))
    print("wrote", path)
