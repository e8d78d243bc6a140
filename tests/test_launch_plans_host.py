"""Rules of the launches that need no device (csrc/plan.h, compiled here with the host compiler), on the CPU."""
import ctypes
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2104_11805_b200", "csrc")

WRAPPER = """
#include "plan.h"
using namespace sdnn_plan;
extern "C" int ctas(int n) { return vector_ctas(n); }
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, lib = d / "plan.cpp", d / "libplan.so"
    src.write_text(WRAPPER)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", "-I", CSRC, "-o", str(lib), str(src)])
    return ctypes.CDLL(str(lib))


class Fault(Exception):
    pass


def exchange(owners, ctas, depth, rng):
    """The exchange of vector_infer_kernel as its comments state it, under a random schedule: `ctas` CTAs run the layers, the first
    `owners` of them have rows and send them.  A CTA's barrier (k % 2) counts layer k: armed for all of the layer, completed when
    `owners` messages are in.  Raises Fault where a message meets a barrier or a buffer that is not ready for it."""
    step = [("send", 0)] * ctas                 # what each CTA does next
    armed = [[1, 0] for _ in range(ctas)]       # layers that each barrier has been armed for (layer 0 before the loop)
    done = [[0, 0] for _ in range(ctas)]        # ... and has completed
    arrived = [[0, 0] for _ in range(ctas)]     # messages of the phase that is open
    read = [-1] * ctas                          # last layer whose inputs the CTA has read
    flying = []                                 # (sender, receiver, layer)

    def settle(r, b):
        if armed[r][b] > done[r][b] and arrived[r][b] == owners:
            done[r][b] += 1
            arrived[r][b] = 0

    slow = rng.randrange(ctas)                  # held back until nothing else can move
    while flying or any(s is not None for s in step):
        moves = [("message", i) for i in range(len(flying))]
        for r in range(ctas):
            if step[r] and (step[r][0] == "send" or done[r][step[r][1] % 2] > step[r][1] // 2):
                moves.append(("cta", r))
        if not moves:
            raise Fault("everybody waits")
        rest = [m for m in moves if m != ("cta", slow)]
        kind, i = rng.choice(rest if rest and rng.random() < 0.98 else moves)
        if kind == "message":
            sender, r, k = flying.pop(i)
            if done[r][k % 2] != k // 2:
                raise Fault("counted on the barrier of layer %d, meant for %d" % (2 * done[r][k % 2] + k % 2, k))
            if read[r] < k - 1:
                raise Fault("layer %d's outputs over inputs still to be read" % k)
            arrived[r][k % 2] += 1
            settle(r, k % 2)
            continue
        what, k = step[i]
        if what == "send":
            read[i] = k
            if i < owners:
                if any(f[0] == i and f[2] == k - 2 for f in flying):
                    raise Fault("layer %d written over a copy under way" % k)
                flying += [(i, r, k) for r in range(ctas)]
            step[i] = ("wait", k)
        else:
            if k + 1 < depth:
                armed[i][(k + 1) % 2] += 1
                settle(i, (k + 1) % 2)
                step[i] = ("send", k + 1)
            else:
                step[i] = None


def test_whole_network_exchange_stays_in_step(plan):
    """Only the CTAs that have rows may take part: with the others waiting along, as a fixed cluster of 16 would have them, nets of
    at most 960 neurons have schedules in which a message meets the wrong phase (the model finds one)."""
    block, cluster = 64, 16
    for n in [1, 63, 64, 65, 128, 600, 959, 960, 961, 1023, 1024, 1025, 2048, 4096]:
        owners = min(cluster, (n + block - 1) // block)
        for seed in range(25):
            exchange(owners, plan.ctas(n), 6, random.Random(seed))
    with pytest.raises(Fault):
        for seed in range(25):
            exchange((600 + block - 1) // block, cluster, 6, random.Random(seed))
