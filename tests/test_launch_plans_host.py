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
extern "C" int cols(int cnt, long long elems, int windows) { return tile_shape(cnt, elems, windows).cols; }
extern "C" int chunk(int cnt, long long elems, int windows) { return tile_shape(cnt, elems, windows).cw; }
extern "C" int graph(int layers, long long elems, int cols, int track) { return tile_as_graph(layers, elems, cols, track); }
extern "C" int rows_log(int n, long long elems, int cw) { return split_rows(n, elems, cw, 148); }
extern "C" int csr(int n, double per_row, int width, int chunks) { const CsrGroups g = csr_groups(n, per_row, width, chunks); return g.groups * 2 + g.narrow; }
extern "C" double row_of(const int64_t* offset, int layers, int l, int n) { return csr_row(offset, layers, l, n); }
extern "C" int call_log(int n, long long elems, int tile) { return call_rows(n, elems, tile, 148); }
extern "C" int shared_chunk(int cnt, long long elems, int ls) { const TileShape t = tile_shape(cnt, elems, false, ls); return t.cw == t.cols ? t.cw : 0; }
extern "C" int asks(long long bytes, int width) { return asks_ahead(bytes, width, 132644864); }
extern "C" int graphs_of_two_orders() {
    GraphKey have[4], want;
    int64_t asked[4] = {1, 0, 0, 0};
    bool make = false;
    have[0].cw = have[0].cols = have[0].used = 16; want = have[0];
    have[0].ls = 2;
    return pick_graph(have, asked, 4, want, make) != 0 && make;
}
extern "C" int units(const int* off, int n, int rows, int bytes, long long slots, int backward, unsigned* out) {
    const std::vector<unsigned> list = split_units(std::vector<int>(off, off + (n + 15) / 16 + 1), n, rows, bytes, 148, slots, backward != 0);
    std::copy(list.begin(), list.end(), out);
    return (int)list.size();
}
extern "C" int graphs_made(const int* cols, const int* used, int calls, int* served_with) {
    GraphKey have[4];
    int64_t asked[4] = {};
    int made = 0;
    for (int i = 0; i < calls; ++i) {
        GraphKey want;
        want.cw = want.cols = cols[i]; want.used = used[i];
        bool make = false;
        const int q = pick_graph(have, asked, 4, want, make);
        if (make) { have[q] = want; ++made; }
        asked[q] = i + 2;
        served_with[i] = have[q].cols == cols[i] ? have[q].used : -1;
    }
    return made;
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, lib = d / "plan.cpp", d / "libplan.so"
    src.write_text(WRAPPER)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", "-I", CSRC, "-o", str(lib), str(src)])
    lib = ctypes.CDLL(str(lib))
    for f in (lib.cols, lib.chunk):
        f.argtypes = [ctypes.c_int, ctypes.c_longlong, ctypes.c_int]
    lib.graph.argtypes = [ctypes.c_int, ctypes.c_longlong, ctypes.c_int, ctypes.c_int]
    return lib


@pytest.mark.parametrize("width", [8, 16, 32, 64, 128])
@pytest.mark.parametrize("n", [1, 15, 16, 17, 700, 1500, 6007])
def test_units_of_layers_that_do_not_fill_the_device(plan, width, n):
    """Every row once, in units within a slice and with as many rows as groups of lanes are left for; no more units than fit; where there
    are units, the longest chain is shorter than it was."""
    plan.units.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_longlong, ctypes.c_int, ctypes.c_void_p]
    rng = random.Random(n * width)
    rows, slices = 32 // (width // 8), (n + 15) // 16
    for steps in ([4] * slices, [rng.randint(0, 7) for _ in range(slices)], sorted((rng.randint(1, 9) for _ in range(slices)), reverse=True), [0] * slices):
        off = [0]
        for s in steps:
            off.append(off[-1] + 128 * s)
        arr, out = (ctypes.c_int * len(off))(*off), (ctypes.c_uint * (32 * slices + 32))()
        for slots in (16, 1184, 2368):
            for backward in (0, 1):
                got = [out[i] for i in range(plan.units(arr, n, rows, 4 * width, slots, backward, out))]
                if not got:
                    continue
                assert len(got) <= slots
                taken, longest = [], 0
                for d in got:
                    row, parts = d >> 3, 1 << (d & 7)
                    assert parts <= rows and row // 16 == (row + rows // parts - 1) // 16
                    taken += [r for r in range(row, row + rows // parts) if r < n]
                    longest = max(longest, -(-steps[row // 16] // parts))
                assert taken == list(range(n)) and longest < max(steps)


def test_rows_shared_in_inference(plan):
    """A group of lanes fits a warp as often as a row is shared, the launch fits the device, and no part of a row is without a step."""
    plan.rows_log.argtypes = [ctypes.c_int, ctypes.c_longlong, ctypes.c_int]
    for n in (1, 17, 700, 1024, 4096, 6007, 16384, 70000):
        for per_row in (0, 8, 32, 56, 300):
            assert plan.rows_log(n, n * per_row, 4) == plan.rows_log(n, n * per_row, 256) == 0
            for cw in (8, 16, 32, 64, 128):
                parts = 1 << plan.rows_log(n, n * per_row, cw)
                assert parts == 1 or (cw // 8 * parts <= 32 and n * (cw // 8) * parts <= 65536 and parts * 8 <= per_row)
    assert plan.rows_log(700, 700 * 32, 64) == 2 and plan.rows_log(16384, 16384 * 32, 64) == 0


def test_rows_of_allocation_free_calls(plan):
    """Groups for every size, none for rows of a few entries; what the offsets say of a row, in any order of the layers, and what they don't."""
    plan.csr.argtypes = [ctypes.c_int, ctypes.c_double, ctypes.c_int, ctypes.c_int]
    plan.row_of.restype = ctypes.c_double
    for n in (1, 17, 700, 1699, 4096, 5121, 9201, 16385, 30000, 262144, 2**31 - 1):
        for width, chunks in [(4, 1), (8, 1), (16, 1), (32, 1), (64, 1), (128, 1), (128, 2), (128, 3), (128, 8192)]:
            for per_row in (0.0, 8.0, 12.0, 24.0, 32.0, 300.0):
                groups = plan.csr(n, per_row, width, chunks) // 2
                assert 0 <= groups <= 8 and (groups >= 4 if width == 4 else groups <= 1 or per_row >= 10)
    assert plan.csr(4096, 32.0, 128, 1) // 2 == 1 and plan.csr(700, 32.0, 128, 1) // 2 == 5 and plan.csr(700, 8.0, 128, 1) // 2 == 1
    offsets = (ctypes.c_int64 * 4)(0, 3200, 6400, 800)
    assert [plan.row_of(offsets, 4, l, 100) for l in range(4)] == [32.0, 32.0, 32.0, 32.0]      # the third layer's end is not known: nor is the fourth's
    offsets = (ctypes.c_int64 * 3)(0, 800, 2**62)
    assert plan.row_of(offsets, 3, 0, 100) == 8.0 and plan.row_of(offsets, 3, 2, 100) > 1e15 and plan.row_of(offsets, 1, 0, 100) == 32.0


def test_the_last_tile_of_a_call_shares_its_rows_like_the_others(plan):
    """Rows are shared by what a call's whole tiles hold.  A narrower last tile keeps to that: one chunk of whole lanes, whose groups fit a
    warp, and a graph of its own where a tile of its width in another call shares rows otherwise."""
    plan.call_log.argtypes = [ctypes.c_int, ctypes.c_longlong, ctypes.c_int]
    plan.shared_chunk.argtypes = [ctypes.c_int, ctypes.c_longlong, ctypes.c_int]
    for n in (17, 700, 1500, 4096, 9000, 30000):
        for per_row in (8, 32, 300):
            for tile in (1, 4, 5, 8, 12, 28, 60, 100, 128, 129, 300):
                ls = plan.call_log(n, n * per_row, tile)
                assert ls == 0 if tile <= 4 or tile > 128 else ls == plan.rows_log(n, n * per_row, plan.cols(tile, n * per_row, 0))
                for last in range(1, tile + 1) if ls else ():
                    cw = plan.shared_chunk(last, n * per_row, ls)
                    assert 8 <= cw <= plan.cols(tile, n * per_row, 0) and cw // 8 << ls <= 32 and last <= cw
    assert plan.call_log(700, 700 * 32, 100) == 1 and plan.call_log(700, 700 * 32, 12) == 2
    assert plan.graphs_of_two_orders()


def test_entries_at_hand_are_not_asked_for(plan):
    """Launches ask for the next one's entries where a pass over the net walks more than stays at hand: a third of L2 in wide train steps,
    all of it in narrow ones, a sixth in inference."""
    plan.asks.argtypes = [ctypes.c_longlong, ctypes.c_int]

    def step(n, layers, width):
        return plan.asks(n * 32 * 12 * layers + 8 * layers * n * width, width)
    assert [step(700, 24, w) for w in (8, 16, 32, 64, 128)] == [0] * 5
    assert step(6007, 56, 64) and step(6007, 24, 64) and step(700, 100, 128) and step(6007, 56, 32) and not step(700, 100, 32) and not step(1500, 100, 16)
    assert not plan.asks(700 * 32 * 6 * 120, 0) and plan.asks(1500 * 32 * 6 * 120, 0)


def test_tile_shapes(plan):
    """Every tile holds its inputs in whole chunks within the widest tile its width stands for; narrow layers keep one chunk; nets with
    their operands in shared memory pad to 32 columns whatever their layers hold."""
    for cnt in list(range(1, 700)) + [1000, 1024, 1025, 4000]:
        widest = plan.cols(cnt, 0, 0)
        for elems in (0, 1 << 15, 1 << 17, 1 << 21, 1 << 28):
            cw, cols = plan.chunk(cnt, elems, 0), plan.cols(cnt, elems, 0)
            assert cnt <= cols <= widest and cols % cw == 0
            if elems * cnt < 32 << 20:
                assert cols == widest
            assert plan.cols(cnt, elems, 1) == (widest if cnt <= 32 else (cnt + 31) // 32 * 32)
    assert plan.cols(300, 131072, 0) == 512 - 192 and plan.cols(150, 524288, 0) == 192


def test_layers_that_outlast_their_launch_call_are_launched_directly(plan):
    """The line is drawn by what a layer holds, at 32 M stored elements x columns, for any layout."""
    assert plan.graph(120, 1 << 17, 256, 0) and not plan.graph(120, (1 << 17) + 1, 256, 0)
    assert plan.graph(120, 1 << 21, 1024, 1) and not plan.graph(3, 1, 4, 0)


def graphs_made(plan, tiles):
    n = len(tiles)
    arrays = [(ctypes.c_int * n)(*[t[q] for t in tiles]) for q in range(2)]
    out = (ctypes.c_int * n)()
    made = plan.graphs_made(*arrays, n, out)
    assert all(used <= got <= cols for (cols, used), got in zip(tiles, out))
    return made, list(out)


def test_graphs_gather_no_more_padding_than_they_have_to(plan):
    """Up to four kinds of tile each have a graph of their own, as wide as their inputs; sizes that vary at will fill the four places and
    then make one per shape; tiles of as many shapes as places settle."""
    kinds = [(128, 72), (128, 104), (256, 136), (8, 8)]
    made, got = graphs_made(plan, kinds * 5)
    assert made == 4 and got == [used for _, used in kinds] * 5
    rng = random.Random(1)
    made, _ = graphs_made(plan, [(128, rng.randrange(72, 129, 8)) for _ in range(500)])
    assert made <= 5
    for shapes in (2, 4):
        tiles = []
        for i in range(2000):
            cols = 64 << i % shapes
            tiles.append((cols, rng.randrange(cols // 2 + 8, cols + 1, 8)))
        early, _ = graphs_made(plan, tiles[:1000])
        assert graphs_made(plan, tiles)[0] == early <= 4 + 2 * shapes


def test_no_kernel_is_given_a_memory_split_for_the_whole_process():
    """The split between L1 and shared memory is asked for launch by launch: set on a kernel it would hold for every handle."""
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            assert "cudaFuncAttributePreferredSharedMemoryCarveout" not in f.read(), name


class Fault(Exception):
    pass


def exchange(owners, ctas, depth, rng, mute=None, careless=False):
    """The exchange of vector_infer_kernel as its comments state it, under a random schedule: `ctas` CTAs run the layers, the first
    `owners` of them have rows and send them.  A CTA's barrier (k % 2) counts layer k: armed for all of the layer, completed when
    `owners` messages are in.  Raises Fault where a message meets a barrier or a buffer that is not ready for it.
    mute: (CTA, layer) whose messages are lost, so that waits run out; careless: a CTA that gave up goes on sending and arming.
    Returns the CTAs that gave up."""
    gave_up = set()
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
            if step[r] and (step[r][0] == "send" or r in gave_up or done[r][step[r][1] % 2] > step[r][1] // 2):
                moves.append(("cta", r))
        if not moves:                           # a wait runs out only where nothing else can happen
            if mute is None:
                raise Fault("everybody waits")
            i = rng.choice([r for r in range(ctas) if step[r]])
            gave_up.add(i)
            moves = [("cta", i)]
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
            if i < owners and (careless or i not in gave_up):
                if any(f[0] == i and f[2] == k - 2 for f in flying):
                    raise Fault("layer %d written over a copy under way" % k)
                flying += [(i, r, k) for r in range(ctas) if (i, k) != mute]
            step[i] = ("wait", k)
        else:
            if k + 1 < depth:
                if careless or i not in gave_up:
                    b = (k + 1) % 2
                    if armed[i][b] > done[i][b]:
                        raise Fault("armed for layer %d with the last phase still open" % (k + 1))
                    armed[i][b] += 1
                    settle(i, b)
                step[i] = ("send", k + 1)
            else:
                step[i] = None
    return gave_up


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


def test_whole_network_exchange_ends_when_a_message_is_lost(plan):
    """A layer's part that never arrives: every CTA that needs it gives up in its turn, and none counts on a barrier again whose
    phase it has not seen the end of (which going on as if nothing had happened would)."""
    for n in [100, 600, 1024]:
        ctas = plan.ctas(n)
        for seed in range(25):
            rng = random.Random(seed)
            lost = (rng.randrange(ctas), rng.randrange(5))
            assert exchange(ctas, ctas, 6, rng, mute=lost) == set(range(ctas))
    with pytest.raises(Fault):
        for seed in range(25):
            exchange(10, 10, 6, random.Random(seed), mute=(3, 2), careless=True)


RESIDENT = """
#include "resident.h"
using namespace sdnn_plan;
extern "C" int width(int n, double elems, long long inputs, int sms, int tile, int drop) { return resident_width(n, elems, inputs, sms, tile, drop != 0); }
extern "C" int layer_width(int n, int chunks, int longest, int several, long long inputs, int tile, int drop) {
    return resident_width(ResidentLayer{n, 4.0 * chunks * n, longest, several != 0}, inputs, 148, tile, drop != 0);
}
extern "C" double cost(int n, int chunks, int longest, int several, long long inputs, int p) {
    return resident_shape(n, p).ok ? resident_clocks(ResidentLayer{n, 4.0 * chunks * n, longest, several != 0}, inputs, 148, p) : 1e30;
}
extern "C" void shape(int n, int p, int* out) {
    const ResidentShape s = resident_shape(n, p);
    out[0] = s.ok; out[1] = s.units; out[2] = s.slots; out[3] = s.cap; out[4] = s.held;
}
extern "C" void share(int total, int sms, int p, int q, int* out) { resident_share(total, sms, p, q, out, out + 1); }
extern "C" int half(int n, long long inputs, int sms) { return resident_half(n, inputs, sms); }
extern "C" int pays(int n, long long inputs, int sms) { return resident_half_pays(n, inputs, sms); }
// steps of a group: left[row][class] entries; read[step][row] = class, 8 + class of the zeros for a row that waits
extern "C" void steps(int* left, int steps, int* read) {
    int total[8] = {};
    for (int r = 0; r < 8; ++r) for (int c = 0; c < 8; ++c) total[c] += left[r * 8 + c];
    for (int t = 0; t < steps; ++t) {
        uint64_t have = 0;
        uint32_t must = 0;
        for (int r = 0; r < 8; ++r) {
            int togo = 0;
            for (int c = 0; c < 8; ++c) { togo += left[r * 8 + c]; if (left[r * 8 + c]) have |= (uint64_t)1 << (8 * c + r); }
            if (togo && togo >= steps - t) must |= 1u << r;
        }
        const uint32_t row = resident_step(have, total, must, steps - t);
        for (int r = 0; r < 8; ++r) {
            const int c = (row >> (4 * r)) & 15;
            read[t * 8 + r] = c == 15 ? 8 + resident_idle_class(row, r) : c;
            if (c != 15) { --left[r * 8 + c]; --total[c]; }
        }
    }
}
"""


@pytest.fixture(scope="module")
def resident(tmp_path_factory):
    d = tmp_path_factory.mktemp("resident")
    src, lib = d / "resident.cpp", d / "libresident.so"
    src.write_text(RESIDENT)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", "-I", CSRC, "-o", str(lib), str(src)])
    lib = ctypes.CDLL(str(lib))
    lib.width.argtypes = [ctypes.c_int, ctypes.c_double, ctypes.c_longlong, ctypes.c_int, ctypes.c_int, ctypes.c_int]
    return lib


def test_shapes_of_networks_held_in_shared_memory(resident):
    """Inputs, free slots and the units held in registers make room for a layer's outputs, within 226 KB; wider needs more room."""
    out = (ctypes.c_int * 5)()
    for n in list(range(1, 300)) + list(range(300, 9000, 37)) + [1024, 2048, 4096, 4608, 4609, 8192, 8193, 20000, 65536]:
        fitted = True
        for p in range(1, 5):
            resident.shape(n, p, out)
            ok, units, slots, cap, held = out
            assert units * 32 >= n > (units - 1) * 32 and slots == units * 32 + 8
            if not ok:
                fitted = False
                continue
            assert fitted and cap * 16 * p <= 226 * 1024 and cap % 8 == 0 and slots <= cap
            rounds = (units + 15) // 16
            assert rounds >= held and (held or cap >= 2 * slots)
            assert min(units, (rounds - held) * 16) * 32 <= cap - slots      # what is stored at once overwrites no input
            assert held <= (4 if p <= 2 else 2)
        if n > 8192:
            assert not fitted and resident.width(n, 32.0 * n, 10000, 148, 1024, 0) == 0


def test_shares_of_networks_held_in_shared_memory(resident):
    """The launches of all widths take every input once; the last round is as narrow as it can be."""
    out = (ctypes.c_int * 2)()
    for sms in (1, 148):
        for p in range(1, 5):
            for total in list(range(0, 60)) + [4 * sms * q + d for q in range(1, 13) for d in (-1, 0, 1)] + [10000, 16384]:
                taken = []
                for q in range(p, 0, -1):
                    resident.share(total, sms, p, q, out)
                    taken += list(range(out[0], out[1]))
                    if q < p:
                        assert out[1] - out[0] <= 4 * q * sms
                assert taken == list(range(total))


def test_halves_of_single_chunks_stay_with_the_layer_launches(resident):
    """Wider nets' halves of up to 256 inputs go through the layer launches, larger ones and those of narrow nets as before."""
    resident.pays.argtypes = resident.half.argtypes = [ctypes.c_int, ctypes.c_longlong, ctypes.c_int]
    for n in (700, 1024, 1025, 2048, 3000, 4000):
        for inputs in (7, 260, 300, 512, 513, 592, 593):
            want = 0 if n > 1024 and inputs <= 512 else resident.half(n, inputs, 148)
            assert resident.pays(n, inputs, 148) == want


def test_widths_of_networks_held_in_shared_memory(resident):
    """The way that was measured to be the faster one (us per layer, layer launches / whole networks), rows of 32 and of 8 to 56 entries; with dead
    inputs dropped a width that is right for all inputs as well as for a third of them."""
    measured = [(700, 32, 300, 300, 4.7, 4.1), (6000, 16, 1500, 1024, 38, 44), (1024, 32, 256, 256, 3.5, 4.8), (1024, 32, 1000, 1000, 8.2, 6.8),
                (4096, 32, 10000, 1024, 269, 208), (8000, 32, 592, 592, 38.4, 34.3), (8000, 32, 1184, 1024, 66.2, 68.7), (5000, 56, 2368, 1024, 134, 147),
                (1024, 0, 592, 592, 8.9, 5.4), (3000, 0, 592, 592, 18.6, 13.7), (7000, 0, 1776, 1024, 89.8, 109), (6000, 0, 2368, 1024, 108, 120), (8000, 0, 592, 592, 39.2, 42.7)]
    resident.layer_width.argtypes = [ctypes.c_int] * 4 + [ctypes.c_longlong, ctypes.c_int, ctypes.c_int]
    resident.cost.argtypes, resident.cost.restype = [ctypes.c_int] * 4 + [ctypes.c_longlong, ctypes.c_int], ctypes.c_double
    for n, k, inputs, tile, launches, whole in measured:
        layer = (n, k // 4, k, 0) if k else (n, 9, 56, 1)
        assert (resident.layer_width(*layer, inputs, tile, 0) > 0) == (whole < launches), (n, k, inputs)
    for n in (640, 1024, 1465, 2048, 4096, 8000):
        for layer in ((n, 4, 16, 0), (n, 8, 32, 0), (n, 9, 56, 1)):
            for inputs in list(range(260, 2400, 37)) + [3000, 5000, 12057, 20000]:
                p = resident.layer_width(*layer, inputs, 1024, 1)
                assert p == 0 or resident.layer_width(*layer, inputs, 1024, 0)
                for left in (inputs, (inputs + 2) // 3) if p else ():
                    assert resident.cost(*layer, left, p) <= 1.06 * min(resident.cost(*layer, left, q) for q in range(1, 5)), (layer, inputs, left)


def test_halves_of_a_batch_from_host_memory(resident):
    """Both halves hold inputs, and their CTAs fit the device side by side."""
    resident.half.argtypes = [ctypes.c_int, ctypes.c_longlong, ctypes.c_int]
    for sms in (4, 148):
        for inputs in range(0, 5 * sms):
            first = resident.half(3000, inputs, sms)
            if first:
                assert 0 < first < inputs and first % 4 == 0 and first // 4 + (inputs - first + 3) // 4 <= sms
            else:
                assert inputs < 8 or inputs > 4 * sms
            assert resident.half(4000, inputs, sms) == 0


@pytest.mark.parametrize("spread", [0, 1, 5])
def test_steps_of_eight_rows(resident, spread):
    """Every entry is read once, in as few wavefronts as the group's counts allow where the rows are of one length (the largest distance of a
    class from the mean on top of one per step); rows that wait read zeros of a class that nobody else reads in that step."""
    rng = random.Random(spread)
    for case in range(200):
        steps = rng.choice([4, 8, 32, 56, 248])
        lens = [max(0, steps - rng.randint(0, spread)) if spread else steps for _ in range(8)]
        skew = rng.choice([1, 1, 1, 4])
        counts = (ctypes.c_int * 64)()
        for r in range(8):
            for _ in range(lens[r]):
                counts[r * 8 + min(rng.randrange(8 * skew), 7)] += 1
        before = list(counts)
        total = [sum(before[c::8]) for c in range(8)]
        read = (ctypes.c_int * (8 * steps))()
        resident.steps(counts, steps, read)
        assert not any(counts)
        waves, seen = 0, [0] * 64
        for t in range(steps):
            row = list(read[t * 8:t * 8 + 8])
            for r, c in enumerate(row):
                if c < 8:
                    seen[r * 8 + c] += 1
            waits = [c - 8 for c in row if c >= 8]
            assert len(set(waits)) == len(waits) and not set(waits) & {c for c in row if c < 8}
            waves += max(row.count(c) for c in set(row))
        assert seen == before
        if not spread and skew == 1:
            assert waves == steps + max(abs(c - steps) for c in total)


CAPTURE_WRAPPER = """
#include "capture.h"
// calls that fail where `which` says so (1 begin, 2 end, 3 a launch, 4 instantiation; 5: the body itself) and note what happened
static int which, open_captures, graphs, execs;
struct Fake {
    using Graph = int;
    int begin() const { if (which == 1) return 100; ++open_captures; return 0; }
    int end(int* g) const { --open_captures; if (which == 2) return 200; ++graphs; *g = 7; return 0; }
    int last_error() const { return which == 3 ? 300 : 0; }
    int instantiate(int* exec, int) const { if (which == 4) return 400; ++execs; *exec = 9; return 0; }
    void destroy(int) const { --graphs; }
};
extern "C" int capture(int fails, int* state) {
    which = fails; open_captures = graphs = execs = 0;
    int exec = 0;
    const int rc = sdnn_plan::capture_graph(Fake{}, &exec, [] { return which == 5 ? -5 : 0; }, [](int e, const char*) { return -e; });
    state[0] = open_captures; state[1] = graphs; state[2] = execs; state[3] = exec;
    return rc;
}
"""


def test_no_graph_is_kept_of_a_capture_that_failed(tmp_path):
    """A capture that was begun is ended, the captured graph is given back, and there is something to launch only if everything went well:
    not where the body gave up, a launch failed, or a call did."""
    src, lib = tmp_path / "capture.cpp", tmp_path / "libcapture.so"
    src.write_text(CAPTURE_WRAPPER)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", "-I", CSRC, "-o", str(lib), str(src)])
    lib = ctypes.CDLL(str(lib))
    state = (ctypes.c_int * 4)()
    for fails, rc in ((0, 0), (1, -100), (2, -200), (3, -300), (4, -400), (5, -5)):
        assert lib.capture(fails, state) == rc
        assert list(state) == ([0, 0, 1, 9] if fails == 0 else [0, 0, 0, 0]), fails
    source = open(os.path.join(CSRC, "sdnn.cu")).read()
    product, probes = source.split('extern "C" int sdnn_probe_gather_rate')[:2]
    assert product.count("cudaStreamBeginCapture(") == product.count("cudaGraphInstantiate(") == 1      # both in what capture_graph is given
    assert "if (const int rc = forward_vector(h, v)) return rc;" in product


def test_a_tile_gives_the_launch_stream_back_wherever_it_returns():
    """The launch helpers' stream is a lane's only while an object lives whose end gives it back; the backward chain sets and clears it around
    launches that do not return."""
    source = open(os.path.join(CSRC, "sdnn.cu")).read()
    tile = source[source.index("\nint infer_tile("):source.index("// Inputs per inference tile.")]
    assert "const LaneScope scope(h, ln);" in tile and "h->launch_stream =" not in tile and "h->cur =" not in tile
    assert source.count("h->launch_stream = ln.stream") == 1 and "~LaneScope() { h->launch_stream = nullptr; h->cur = &h->lane[0]; }" in source
