"""The wait order of the kernels' pipelines (csrc/pipeline.h), run on the host: barriers as the hardware has them -- a phase
completes after its count of arrivals, and a wait names a phase by its parity alone -- and roles that wait for one another as
the kernels' warps do, at many timings.  A role that misses a phase waits for ever; here that ends the run with an error."""
import ctypes
import heapq
import os
import random
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_20488_b200", "csrc")

SHIM = r"""
#include "pipeline.h"
using namespace firp;
extern "C" {
int kv_ring() { return kRowsKvRing; }
int spo_ring() { return kRowsSpoRing; }
int kv_bar(int i) { return rows_kv(i).bar; }
int kv_parity(int i) { return rows_kv(i).parity; }
int spo_bar(int i) { return rows_spo(i).bar; }
int spo_parity(int i) { return rows_spo(i).parity; }
typedef int (*Free)(int, int, unsigned);
typedef void (*Load)(int, int);
typedef void (*Landed)(int, unsigned);
struct Ring {
  Free f; Load l; Landed d;
  bool free(int u, int slot, unsigned parity) { return f(u, slot, parity) != 0; }
  void load(int u, int slot) { l(u, slot); }
  void landed(int slot, unsigned parity) { d(slot, parity); }
};
void run_producer(int n, int depth, Free f, Load l, Landed d) { Ring r{f, l, d}; drain(r, produce(r, n, depth), depth); }
}
"""


@pytest.fixture(scope="module")
def order(tmp_path_factory):
    d = tmp_path_factory.mktemp("pipeline")
    src = d / "shim.cpp"
    src.write_text(SHIM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "shim.so"), str(src)])
    return ctypes.CDLL(str(d / "shim.so"))


class Barrier:
    def __init__(self, count):
        self.count, self.pending, self.done = count, count, 0

    def arrive(self):
        self.pending -= 1
        if self.pending == 0:
            self.pending, self.done = self.count, self.done + 1

    def complete(self, parity):        # the phase of that parity: the one before the current one
        return (self.done & 1) != parity


def simulate(roles):
    """roles: generators that yield ("wait", barrier, parity), ("busy", time) or ("later", time, barrier): an arrival then.
    Returns the names of the roles that are still waiting when nothing is left to happen."""
    events, waiting, n, now = [], [], 0, 0.0
    ready = [(name, g) for name, g in roles]
    while True:
        while ready:
            name, g = ready.pop()
            for op in g:
                if op[0] == "wait":
                    if not op[1].complete(op[2]):
                        waiting.append((name, g, op[1], op[2]))
                        break
                elif op[0] == "busy":
                    heapq.heappush(events, (now + op[1], n, None, (name, g)))
                    n += 1
                    break
                else:
                    heapq.heappush(events, (now + op[1], n, op[2], None))
                    n += 1
        if not events:
            return [w[0] for w in waiting]
        now, _, bar, role = heapq.heappop(events)
        if bar is not None:
            bar.arrive()
        else:
            ready.append(role)
        still = []
        for w in waiting:
            (ready.append((w[0], w[1])) if w[2].complete(w[3]) else still.append(w))
        waiting = still


def attention_roles(order, ntiles, load, softmax, mma, output):
    """The roles of tree_attn_rows_kernel (attn_tc.cu); load(is_v, i), softmax(i), mma(), output() give times."""
    kvr, spr = order.kv_ring(), order.spo_ring()
    full = {v: [Barrier(1) for _ in range(kvr)] for v in (0, 1)}
    s, p, o = ([Barrier(1) for _ in range(spr)] for _ in range(3))
    o_free = Barrier(1)
    handed = [Barrier(1) for _ in range(ntiles + 1)]        # the running maximum, from tile to tile

    def of(ring, i):
        return "wait", ring[order.spo_bar(i)], order.spo_parity(i)

    def of_kv(v, i):
        return "wait", full[v][order.kv_bar(i)], order.kv_parity(i)

    def producer(v):
        for i in range(ntiles):
            if i >= kvr:
                yield of(o if v else s, i - kvr)
            yield "later", load(v, i), full[v][order.kv_bar(i)]

    def issue_s():
        for i in range(ntiles):
            yield of_kv(0, i)
            if i >= spr:
                yield of(o, i - spr)
            yield "later", mma(), s[order.spo_bar(i)]

    def issue_o():
        for i in range(ntiles):
            yield of_kv(1, i)
            if i >= 1:
                yield "wait", o_free, (i - 1) & 1
            yield of(p, i)
            yield "later", mma(), o[order.spo_bar(i)]

    def soft(g):
        for i in range(g, ntiles, 2):
            yield of(s, i)
            yield "busy", softmax(i) / 2
            if i > 0:
                yield "wait", handed[i], 0
            handed[i + 1].arrive()
            yield "busy", softmax(i) / 2
            p[order.spo_bar(i)].arrive()
            yield "busy", 0.0

    def out():
        for i in range(ntiles):
            yield of(o, i)
            yield "busy", output()
            o_free.arrive()
            yield "busy", 0.0

    return [("K producer", producer(0)), ("V producer", producer(1)), ("S issuer", issue_s()), ("O issuer", issue_o()),
            ("softmax 0", soft(0)), ("softmax 1", soft(1)), ("output", out())]


@pytest.mark.parametrize("v", [0, 1])
@pytest.mark.parametrize("late", range(12))
def test_rows_attention_with_one_late_tile(order, late, v):
    """One K or V tile lands later than everything that does not depend on it takes."""
    for extra in (3.0, 6.0, 50.0):
        stuck = simulate(attention_roles(order, 16, lambda is_v, i: 1.0 + (extra if (is_v, i) == (v, late) else 0.0), lambda i: 2.2, lambda: 0.5, lambda: 0.4))
        assert not stuck, "tile %d %.0f us late: %s" % (late, extra, stuck)


@pytest.mark.parametrize("seed", range(60))
def test_rows_attention_at_random_timings(order, seed):
    rng = random.Random(seed)
    slow = [rng.choice((0.1, 1.0, 10.0)) for _ in range(4)]
    stuck = simulate(attention_roles(order, rng.randint(1, 24), lambda is_v, i: rng.expovariate(1 / slow[0]), lambda i: rng.expovariate(1 / slow[1]),
                                     lambda: rng.expovariate(1 / slow[2]), lambda: rng.expovariate(1 / slow[3])))
    assert not stuck, stuck


@pytest.mark.parametrize("depth", [1, 2, 3, 12])
@pytest.mark.parametrize("n,stops_at", [(0, 99), (1, 99), (2, 99), (5, 99), (13, 99), (40, 99), (40, 0), (40, 1), (40, 3), (40, 11), (40, 12), (40, 25)])
def test_producer_leaves_nothing_in_flight(order, depth, n, stops_at):
    """Loads go in order, each into a slot whose last load its reader has given back, none after a wait that ran out, and every
    one has been seen to land after the drain.  From unit `stops_at` on the readers give no slot back."""
    in_flight, loaded, ran_out, landed = {}, [], [], [0] * depth

    def free(u, slot, parity):
        assert not ran_out and u == len(loaded) and slot == u % depth
        released = u // depth                               # phases that the slot's readers complete for this load, if they do
        assert parity == (released & 1) ^ 1                 # the phase just before: complete at the start, then once per turn
        if u - depth >= stops_at:
            ran_out.append(u)
            return 0
        if u >= depth:                                      # given back: its reader has seen it land
            assert in_flight.pop(slot) == u - depth
            landed[slot] += 1
        return 1

    def load(u, slot):
        assert not ran_out and slot not in in_flight
        loaded.append(u)
        in_flight[slot] = u

    def land(slot, parity):
        assert parity == landed[slot] & 1
        del in_flight[slot]
        landed[slot] += 1

    types = (ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_uint), ctypes.CFUNCTYPE(None, ctypes.c_int, ctypes.c_int),
             ctypes.CFUNCTYPE(None, ctypes.c_int, ctypes.c_uint))
    order.run_producer(n, depth, *(t(f) for t, f in zip(types, (free, load, land))))
    assert not in_flight
    assert loaded == list(range(min(n, stops_at + depth)))
