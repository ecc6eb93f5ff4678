"""The order of waits, issues and slot reuse in the kernels that couple warps by
mbarriers with the labels side by side, replayed on the host under random
schedules in which any one warp may be far slower than the others: no warp ever
waits for a phase that cannot come, and no slot is rewritten while it is read.

The rules (which row is issued when, who waits for what) are the kernels' own,
from csrc/cmf_rows_order.cuh; the replay adds what the kernels do between them."""
import ctypes
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
EXPORTS = """
#include "cmf_rows_order.cuh"
using namespace cmf;
extern "C" {
int state_rows() { return rows::kState; }
int aux_rows() { return rows::kAux; }
int share_rows() { return rows::kSh; }
int ps_rows() { return rows::kPs; }
int service_warps(int T, int LC) { return rows::service_warps(T, LC); }
int issued_after(int k) { return rows::issued_after(k); }
int label_waits_row(int k, int il) { return rows::label_waits_row(k, il); }
int last_input_step(int il) { return rows::last_input_step(il); }
int cert_ring() { return cert::kRing; }
int theta_warps(int LC) { return cert::theta_warps(LC); }
int thresholds_from(int k) { return cert::thresholds_from(k); }
}
"""


@pytest.fixture(scope="module")
def order(tmp_path_factory):
    d = tmp_path_factory.mktemp("order")
    src, so = d / "order.cpp", d / "order.so"
    src.write_text(EXPORTS)
    subprocess.check_call(["g++", "-std=c++17", "-shared", "-fPIC", "-I",
                           os.path.join(ROOT, "paper_2004_11227_gb300", "csrc"), str(src), "-o",
                           str(so)])
    return ctypes.CDLL(str(so))


class Bar:
    """An mbarrier: waits see the parity of the phase last completed only."""

    def __init__(self, count):
        self.count, self.left, self.done = count, count, 0

    def arrive(self):
        self.left -= 1
        assert self.left >= 0, "an arrival too many"
        if self.left == 0:
            self.left, self.done = self.count, self.done + 1

    def passes(self, parity):
        return (self.done - 1) & 1 == parity & 1


def replay(tasks, flight, land, rng, slow, weight):
    """Run the tasks (generators yielding the (barrier, parity) they wait for, or
    None) in a random order, task `slow` picked `weight` times as often as the
    others; True when all of them finish."""
    waiting = [None] * len(tasks)
    alive = list(range(len(tasks)))
    w = [weight if i == slow else 1.0 for i in range(len(tasks) + 1)]
    while alive or flight:
        ready = [i for i in alive if waiting[i] is None or waiting[i][0].passes(waiting[i][1])]
        if flight:
            ready.append(len(tasks))
        if not ready:
            return False
        i = rng.choices(ready, [w[j] for j in ready])[0]
        if i == len(tasks):
            land(flight.pop(rng.randrange(len(flight))))
            continue
        try:
            waiting[i] = next(tasks[i])
        except StopIteration:
            alive.remove(i)
    return True


def admm_rows(o, T, LC, L, n, rng, slow, weight):
    """k_potts_rows: a band of n rows, T iterations, L labels in a class of LC."""
    kS, kA, kSh, kPs = o.state_rows(), o.aux_rows(), o.share_rows(), o.ps_rows()
    il, ke = (n + 4, n + 4) if T == 2 else (n + 2, n)
    full = [Bar(1) for _ in range(kA)]
    sf = [Bar(L) for _ in range(4)]
    pr = [Bar(1) for _ in range(4)]
    pr[0].arrive(), pr[1].arrive()
    state, aux, ps, flight = [None] * kS, [None] * kA, [None] * kPs, []
    sha = [[None] * L for _ in range(kSh)]
    shb = [[None] * L for _ in range(kSh)]
    two = o.service_warps(T, LC) == 2

    def issue(i):
        if i <= il:
            state[i % kS] = aux[i % kA] = "in flight"
            flight.append(i)

    def land(i):
        state[i % kS] = aux[i % kA] = i
        full[i % kA].arrive()

    def service(sums, inputs):
        issued = 0
        while inputs and issued < kS:
            issue(issued)
            issued += 1
            yield None
        for k in range((ke if sums else o.last_input_step(il)) + 1):
            yield sf[k & 3], (k >> 2) & 1
            if sums:
                p_s = aux[(k + 1) % kA]  # of a row behind the last one: not used
                assert k + 1 > il or p_s == k + 1
                yield None
                assert sha[k % kSh] == [k] * L and aux[(k + 1) % kA] == p_s
                if T == 2:
                    ps[k % kPs] = k
                    pr[(k + 2) & 3].arrive()
                    yield None
                    if k >= 4:
                        assert shb[(k - 3) % kSh] == [k - 3] * L and ps[(k - 3) % kPs] == k - 3
            while inputs and issued < o.issued_after(k):
                issue(issued)
                issued += 1
                yield None

    def label(l):
        for i in (0, 1):
            yield full[i], 0
        assert state[0] == 0 and state[1] == 1
        for k in range(ke + 1):
            if o.label_waits_row(k, il):
                yield full[(k + 2) % kA], ((k + 2) // kA) & 1
            if T == 2:
                yield pr[k & 3], (k >> 2) & 1
                if k >= 2:  # p_s, costs and alpha of stage B
                    assert ps[(k - 2) % kPs] == k - 2 and aux[(k - 2) % kA] == k - 2
                yield None
                shb[(k - 3) % kSh][l] = k - 3
            if k + 2 <= il:
                assert state[(k + 2) % kS] == k + 2 and aux[(k + 2) % kA] == k + 2
                yield None
                assert state[(k + 2) % kS] == k + 2
            assert k + 1 > il or aux[(k + 1) % kA] == k + 1
            sha[k % kSh][l] = k
            yield None
            sf[k & 3].arrive()

    tasks = [label(l) for l in range(L)]
    tasks += [service(True, False), service(False, True)] if two else [service(True, True)]
    return replay(tasks, flight, land, rng, slow % (len(tasks) + 1), weight)


@pytest.mark.parametrize("weight", [1.0, 0.1, 0.01, 0.001])
@pytest.mark.parametrize("T,LC,L", [(1, 4, 3), (1, 8, 5), (2, 4, 4), (2, 8, 5), (2, 16, 9)])
def test_admm_rows_never_stuck(order, T, LC, L, weight):
    for n in (1, 2, 3, 5, 9, 20):
        for slow in range(L + 3):
            for seed in range(3):
                assert admm_rows(order, T, LC, L, n, random.Random(seed), slow, weight), \
                    (n, slow, seed)


def certificate_rows(o, LC, L, n, rng, slow, weight):
    """k_potts_cert: a band of n rows, L labels in a class of LC."""
    R, NT = o.cert_ring(), o.theta_warps(LC)
    il, ke = n + 1, n
    full, th = [Bar(1) for _ in range(R)], [Bar(1) for _ in range(R)]
    sf = [Bar(L) for _ in range(R)]
    rows, thr, flight = [None] * R, [None] * R, []
    shares = [[None] * L for _ in range(R)]

    def issue(i):
        if i <= il:
            rows[i % R] = "in flight"
            flight.append(i)

    def land(i):
        rows[i % R] = i
        full[i % R].arrive()

    def label(l):
        yield full[0], 0
        for i in range(o.thresholds_from(0), 1):
            yield th[i], 0
        assert rows[0] == 0
        for k in range(ke + 1):
            yield full[(k + 1) % R], (k + 1) // R & 1
            for i in range(max(1, o.thresholds_from(k)), k + 2):
                yield th[i % R], i // R & 1
            assert rows[(k + 1) % R] == k + 1 and rows[k % R] == k and thr[(k + 1) % R] == k + 1
            yield None
            assert rows[(k + 1) % R] == k + 1 and rows[k % R] == k and thr[(k + 1) % R] == k + 1
            shares[k % R][l] = k
            yield None
            sf[k % R].arrive()

    def theta(w):
        for i in range(w, il + 1, NT):
            yield full[i % R], i // R & 1
            for _ in range(3):
                assert rows[i % R] == i, "overwritten while read"
                yield None
            thr[i % R] = i
            th[i % R].arrive()

    def last():
        for i in range(R):
            issue(i)
            yield None
        for k in range(ke + 1):
            yield sf[k % R], k // R & 1
            assert shares[k % R] == [k] * L
            yield None
            issue(k + R)

    tasks = [label(l) for l in range(L)] + [theta(w) for w in range(NT)] + [last()]
    return replay(tasks, flight, land, rng, slow % (len(tasks) + 1), weight)


@pytest.mark.parametrize("weight", [1.0, 0.1, 0.01, 0.001])
@pytest.mark.parametrize("LC,L", [(4, 3), (8, 5), (16, 9)])
def test_certificate_rows_never_stuck(order, LC, L, weight):
    for n in (1, 2, 6, 7, 8, 9, 20):
        for slow in range(L + LC // 4 + 2):
            for seed in range(3):
                assert certificate_rows(order, LC, L, n, random.Random(seed), slow, weight), \
                    (n, slow, seed)
