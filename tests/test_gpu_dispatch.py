"""Edges of the launch and layout rules (run with -m gpu on a B200): the sizes at which a rule switches, remainders, the
smallest and largest nets of a rule's range, each against the float64 oracle."""
import numpy as np
import pytest

from oracle import OracleNet
from parity_util import check_close, ragged_net
from test_gpu_parity import BWD_MODES, infer_parity, sdnn, torch_cuda, train_parity  # noqa: F401

pytestmark = pytest.mark.gpu


def vectors(rng, count, n):
    return rng.uniform(0, 1.0, size=(count, n)).astype(np.float32)


@pytest.mark.parametrize("n", [1023, 1024, 1041, 2100])
@pytest.mark.parametrize("B", [2, 20])
def test_ragged_rows_stored_by_length(torch_cuda, n, B):  # noqa: F811
    """Rows are sorted by length in blocks of 1024: a block short by one row, a whole one, a second block of one slice and
    one row, a third of a few slices; weights and biases keep the caller's order."""
    rng = np.random.default_rng(n + B)
    arrays = ragged_net(rng, n=n, layers=3, kmax=40, scale=0.3)
    train_parity(torch_cuda, arrays, [(vectors(rng, B, n), vectors(rng, B, n)) for _ in range(2)], eta=0.02, update_bias=True,
                 activation="sigmoid", expect_live=True)
    infer_parity(torch_cuda, arrays, vectors(rng, 3 * B, n), 2 * B, expect_nonempty=True)


@pytest.mark.parametrize("n,k,B", [(4097, 48, 100), (1500, 300, 33), (8200, 32, 33), (16400, 140, 33)])
def test_row_major_copy_moved_from_the_transposed_one(torch_cuda, n, k, B):  # noqa: F811
    """Layers large enough to have their row-major copy filled from the transposed one after an update (blocks of 2048 to
    8192 elements, up to 300 of them, the last one partial, ragged rows and columns), two steps of one handle at the full batch and one at a batch
    narrow enough for row units, against the oracle; both copies hold the same bits."""
    torch, pkg = torch_cuda, sdnn()
    rng = np.random.default_rng(n)
    rps, cols, vals, biases = [], [], [], []
    for _ in range(2):
        length = rng.integers(0, 2 * k, size=n)
        rp = np.zeros(n + 1, dtype=np.int32)
        rp[1:] = np.cumsum(length)
        cols.append(np.concatenate([np.sort(rng.choice(n, size=m, replace=False)) for m in length]).astype(np.int32))
        rps.append(rp)
        vals.append((rng.standard_normal(rp[-1]) * 0.1).astype(np.float32))
        biases.append((rng.standard_normal(n) * 0.1).astype(np.float32))
    h = pkg.Sdnn.create(rps, cols, vals, biases, max_batch=B, train=True, update_bias=True, activation=pkg.ACT_SIGMOID)
    ora = OracleNet(rps, cols, vals, biases, update_bias=True, activation="sigmoid")
    for b in (B, B, 5):
        ora.quantize_state()
        for l in range(2):
            h.set_weights(l, ora.w[l], ora.bias[l])
        x0, y = vectors(rng, b, n), vectors(rng, b, n)
        h.train_step(torch.from_numpy(x0).cuda(), torch.from_numpy(y).cuda(), b, 0.5)
        ora.train_step(x0, y, 0.5, keep=())
        for l in range(2):
            w, bias = h.get_weights(l)
            check_close(w, ora.w[l], f"W^{l + 1} at B = {b}")
            check_close(bias, ora.bias[l], f"b^{l + 1} at B = {b}")
            assert h.mirror_mismatches(l) == 0
    h.destroy()


def uniform_net(rng, n, k, layers):
    """Layers of k entries per row anywhere, made quickly."""
    cols = [(np.sort(rng.integers(0, n - k + 1, size=(n, k)), axis=1) + np.arange(k)).astype(np.int32).ravel() for _ in range(layers)]
    vals = [rng.uniform(-1, 1, size=n * k).astype(np.float32) for _ in range(layers)]
    return [np.arange(n + 1, dtype=np.int32) * k] * layers, cols, vals, [np.zeros(n, dtype=np.float32)] * layers


@pytest.fixture
def all_but(torch_cuda):  # noqa: F811
    """all_but(bytes): takes the device's free memory but for so many bytes until the test is over."""
    torch, held = torch_cuda, []

    def take(room):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        held.append(torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda"))
    yield take
    held.clear()
    torch.cuda.empty_cache()


def test_small_arrays_take_what_is_left(torch_cuda, all_but):  # noqa: F811
    """Small arrays are cut from blocks that double: with less left than the next block, a handle that fits is made all the same."""
    torch, pkg = torch_cuda, sdnn()
    rng = np.random.default_rng(0)
    arrays = uniform_net(rng, 4096, 32, 80)                       # 0.79 MB a layer: blocks of 2, 4, .. 32 MB, then 64 MB for the last few layers
    x = torch.from_numpy(vectors(rng, 8, 4096)).cuda()
    outs, taken = [torch.zeros(8, 4096, device="cuda") for _ in range(2)], []
    for y in outs:
        if taken:
            all_but(72 << 20)
        h = pkg.Sdnn.create(*arrays, max_batch=8, activation=pkg.ACT_SIGMOID)
        h.infer_batch(x, 8, y)
        torch.cuda.synchronize()
        taken.append(h.device_bytes())
        h.destroy()
    assert taken[1] <= 72 << 20 < taken[0]
    assert torch.equal(outs[0], outs[1])


def test_a_training_net_that_just_fits_does_without_the_move_maps(torch_cuda, all_but):  # noqa: F811
    """With room for the net but not for the maps that move its row-major values (60 MB here), row units update them: the same
    launches as for a narrow batch, and the same bits."""
    torch, pkg = torch_cuda, sdnn()
    rng = np.random.default_rng(1)
    n, layers, B = 16384, 24, 64
    arrays = uniform_net(rng, n, 32, layers)
    x, y = (torch.from_numpy(vectors(rng, B, n)).cuda() for _ in range(2))
    taken, launches, weights = [], [], []
    for _ in range(2):
        if taken:
            all_but(taken[0] - (30 << 20))
        h = pkg.Sdnn.create(*arrays, max_batch=B, train=True, activation=pkg.ACT_SIGMOID)
        taken.append(h.device_bytes())
        h.train_step(x, y, B, 0.5)
        launches.append(h.kernel_launches())
        weights.append([h.get_weights(l, want_bias=False) for l in range(layers)])
        assert h.mirror_mismatches(layers - 1) == 0
        h.destroy()
    assert taken[1] <= taken[0] - (50 << 20) and launches[1] == launches[0] - (layers - 1)
    assert all(np.array_equal(a, b) for a, b in zip(*weights))


def test_weights_of_several_handles_read_from_several_threads(torch_cuda):  # noqa: F811
    """Handles share the pinned pieces that weights travel through: small layers, layers of several pieces and biases, read by a thread
    per handle, while handles come and go."""
    from concurrent.futures import ThreadPoolExecutor
    pkg = sdnn()

    def one(seed):
        rng = np.random.default_rng(seed)
        n, k = ((700, 16), (9000, 100), (30000, 61), (4096, 32))[seed % 4]
        rp, cols, vals, _ = uniform_net(rng, n, k, 2)
        bias = [rng.standard_normal(n).astype(np.float32) for _ in range(2)]
        for _ in range(3):
            h = pkg.Sdnn.create(rp, cols, vals, bias, max_batch=4)
            for _ in range(4):
                for l in range(2):
                    w, b = h.get_weights(l)
                    assert np.array_equal(w, vals[l]) and np.array_equal(b, bias[l])
            h.destroy()
        return True
    with ThreadPoolExecutor(4) as pool:
        assert all(pool.map(one, range(8)))


@pytest.mark.parametrize("n,k,layers", [(9, 3, 2), (64, 5, 3), (1000, 32, 4), (1024, 33, 9), (1025, 32, 5), (2047, 8, 12), (4096, 16, 3)])
@pytest.mark.parametrize("cnt", [1, 2, 3])
@pytest.mark.parametrize("act", ["clamped_relu", "sigmoid"])
def test_whole_network_launch(torch_cuda, n, k, layers, cnt, act):  # noqa: F811
    """One to four inputs through a net whose rows all have the same length: a block of 64 rows per CTA and one or more, the
    last one partial or empty, fewer rows than CTAs, rows of more than 32 entries, more layers than the ring of entries has
    stages; twice, so that the second call meets what the first one left."""
    torch, pkg = torch_cuda, sdnn()
    rng = np.random.default_rng(n + k)
    rp = [np.arange(n + 1, dtype=np.int32) * k] * layers
    cols = [np.concatenate([np.sort(rng.choice(n, size=k, replace=False)) for _ in range(n)]).astype(np.int32) for _ in range(layers)]
    vals = [(rng.standard_normal(n * k) * (2.0 / k) ** 0.5).astype(np.float32) for _ in range(layers)]
    bias = [(rng.standard_normal(n) * 0.1).astype(np.float32) for _ in range(layers)]
    h = pkg.Sdnn.create(rp, cols, vals, bias, max_batch=64, activation=pkg.ACT_SIGMOID if act == "sigmoid" else pkg.ACT_CLAMPED_RELU)
    ora = OracleNet(rp, cols, vals, bias, activation=act)
    for _ in range(2):
        x0 = vectors(rng, cnt, n)
        y = torch.full((cnt, n), -1.0, device="cuda")
        c = torch.full((cnt,), -1, dtype=torch.int32, device="cuda")
        before = h.kernel_launches()
        h.infer_batch(torch.from_numpy(x0).cuda(), cnt, y, c)
        torch.cuda.synchronize()
        assert (h.kernel_launches() - before == 1) == (n * (cnt if cnt <= 2 else 4) <= 4096)
        check_close(y.cpu().numpy(), ora.infer(x0), "x^L")
        assert np.array_equal(c.cpu().numpy(), np.count_nonzero(y.cpu().numpy(), axis=1))
    h.destroy()


@pytest.mark.parametrize("n,layers", [(40, 120), (600, 120), (960, 40), (961, 40)])
@pytest.mark.parametrize("cnt", [1, 2, 4])
def test_whole_network_launch_with_ctas_that_have_no_rows(torch_cuda, n, layers, cnt):  # noqa: F811
    """Nets of at most 960 neurons leave some CTAs of the cluster without rows; deep enough, and called often enough, that a CTA
    that got ahead of the others would be noticed: every call the same bits, and the oracle's numbers.  Training runs its forward chain
    the same way."""
    torch, pkg = torch_cuda, sdnn()
    rng = np.random.default_rng(n + cnt)
    k = 32
    rp = [np.arange(n + 1, dtype=np.int32) * k] * layers
    cols = [np.concatenate([np.sort(rng.choice(n, size=k, replace=False)) for _ in range(n)]).astype(np.int32) for _ in range(layers)]
    vals = [rng.uniform(-1, 1, size=n * k).astype(np.float32) for _ in range(layers)]
    bias = [(rng.standard_normal(n) * 0.1).astype(np.float32) for _ in range(layers)]
    x0 = vectors(rng, cnt, n)
    want = OracleNet(rp, cols, vals, bias, activation="sigmoid").infer(x0)
    for train in (False, True):
        h = pkg.Sdnn.create(rp, cols, vals, bias, max_batch=4, train=train, activation=pkg.ACT_SIGMOID)
        x, outs = torch.from_numpy(x0).cuda(), []
        for _ in range(50):
            if train:
                h.train_step(x, torch.zeros_like(x), cnt, 0.0)      # a step of no length: only the activations matter here
            else:
                outs.append(torch.full((cnt, n), -1.0, device="cuda"))
                h.infer_batch(x, cnt, outs[-1])
        got = h.get_activations(layers, cnt) if train else outs[0].cpu().numpy()
        check_close(got, want, "x^L")
        assert all(torch.equal(y, outs[0]) for y in outs)
        h.destroy()


def test_a_wait_that_ran_out_is_reported_by_the_next_call_that_looks(torch_cuda):  # noqa: F811
    """The word that a whole-network launch raises, raised from the host: every call that launches such work or waits for the stream
    reports it, once; sdnn_set_weights leaves the weights as they are; handles without such launches have no word."""
    torch, pkg = torch_cuda, sdnn()
    rng = np.random.default_rng(3)
    n, k, layers = 600, 16, 3
    arrays = ([np.arange(n + 1, dtype=np.int32) * k] * layers,
              [np.concatenate([np.sort(rng.choice(n, size=k, replace=False)) for _ in range(n)]).astype(np.int32)] * layers,
              [(rng.standard_normal(n * k) * 0.3).astype(np.float32)] * layers, [np.zeros(n, dtype=np.float32)] * layers)
    h = pkg.Sdnn.create(*arrays, max_batch=4, train=True, activation=pkg.ACT_SIGMOID, flags=pkg.FLAG_KEEP_DEBUG)
    x0 = vectors(rng, 4, n)
    x, y, host_y, ids = torch.from_numpy(x0).cuda(), torch.zeros(4, n, device="cuda"), np.zeros((4, n), np.float32), torch.zeros(4 * n, dtype=torch.int32, device="cuda")
    h.train_step(x, x, 4, 0.1, want_loss=True)
    kept = h.get_weights(1)
    calls = {
        "train_step": lambda: h.train_step(x, x, 2, 0.1), "train_step with its loss": lambda: h.train_step(x, x, 2, 0.1, want_loss=True),
        "train_step_averaged": lambda: h.train_step(x, x, 4, 0.1, averaged=True), "train_step_host": lambda: h.train_step(x0, x0, 2, 0.1, host=True),
        "infer_batch": lambda: h.infer_batch(x, 1, y), "infer_batch with ids": lambda: h.infer_batch(x, 4, y, None, ids, 4 * n, want_total=True),
        "infer_batch of a tile": lambda: h.infer_batch(x, 4, y, want_total=True), "infer_batch_host": lambda: h.infer_batch(x0, 4, host_y, host=True),
        "get_weights": lambda: h.get_weights(0), "values alone": lambda: h.get_weights(0, want_bias=False),
        "set_weights": lambda: h.set_weights(1, np.ones_like(kept[0]), np.ones_like(kept[1])), "get_activations": lambda: h.get_activations(1, 4),
        "get_delta": lambda: h.get_delta(1, 4), "get_gradient": lambda: h.get_gradient(1), "mirror_mismatches": lambda: h.mirror_mismatches(1),
        "get_phase_times": h.get_phase_times}
    for name, call in calls.items():
        before = h.get_weights(1)
        h.inject_wait_failure()
        with pytest.raises(pkg.SdnnError) as e:
            call()
        assert e.value.code == -4 and "gave up" in e.value.message, name
        if name == "set_weights":
            assert all(np.array_equal(a, b) for a, b in zip(h.get_weights(1), before))
        call()                                                  # reported once
    h.destroy()
    h = pkg.Sdnn.create(*ragged_net(rng, n=n, layers=2, kmax=40, scale=0.3), max_batch=4)
    with pytest.raises(pkg.SdnnError) as e:
        h.inject_wait_failure()
    assert e.value.code == -5
    h.destroy()


@pytest.mark.parametrize("cnt", [65, 129, 150, 300, 449, 513])
def test_tile_widths_between_powers_of_two(torch_cuda, cnt):  # noqa: F811
    """Layers large enough for tiles cut into chunks of 64 or 128 inputs: widths just above a chunk, a few chunks, and one that
    keeps chunks of 256; outputs, counts and id lists."""
    rng = np.random.default_rng(cnt)
    n, k = 8200, 64
    cols = [np.concatenate([np.sort(rng.integers(0, n - k + 1, size=k)) + np.arange(k) for _ in range(n)]).astype(np.int32) for _ in range(2)]
    vals = [(rng.standard_normal(n * k) * (2.0 / k) ** 0.5).astype(np.float32) for _ in range(2)]
    arrays = ([np.arange(n + 1, dtype=np.int32) * k] * 2, cols, vals, [np.zeros(n, dtype=np.float32)] * 2)
    infer_parity(torch_cuda, arrays, vectors(rng, cnt, n), 600, expect_nonempty=True)


@pytest.mark.parametrize("cnt", [255, 256, 300, 500])
def test_host_batches_cut_in_two(torch_cuda, cnt):  # noqa: F811
    """Host batches of one tile around the size from which they are halved: outputs, counts and ids in the order of the inputs."""
    rng = np.random.default_rng(cnt)
    arrays = ragged_net(rng, n=2111, layers=3, kmax=40, scale=0.3)
    infer_parity(torch_cuda, arrays, vectors(rng, cnt, 2111), 512, host=True, expect_nonempty=True)


@pytest.mark.parametrize("n,k,B", [(33, 7, 4), (1000, 32, 1), (1024, 32, 2), (1030, 40, 1), (2047, 16, 1)])
def test_train_with_the_forward_chain_in_one_launch(torch_cuda, n, k, B):  # noqa: F811
    """Narrow nets with rows of one length, up to four inputs: everything a step leaves behind against the oracle, ending with a
    smaller batch of the same padded width, which takes another variant of the launch."""
    rng = np.random.default_rng(n + B)
    cols = [np.concatenate([np.sort(rng.choice(n, size=k, replace=False)) for _ in range(n)]).astype(np.int32) for _ in range(3)]
    vals = [rng.uniform(-1, 1, size=n * k).astype(np.float32) for _ in range(3)]
    arrays = ([np.arange(n + 1, dtype=np.int32) * k] * 3, cols, vals, [(rng.standard_normal(n) * 0.1).astype(np.float32)] * 3)
    batches = [(vectors(rng, B, n), vectors(rng, B, n)) for _ in range(2)]
    train_parity(torch_cuda, arrays, batches, eta=0.02, update_bias=True, activation="sigmoid", expect_live=True)
    torch, pkg = torch_cuda, sdnn()
    h = pkg.Sdnn.create(*arrays, max_batch=4, train=True, activation=pkg.ACT_SIGMOID)
    ora = OracleNet(*arrays, activation="sigmoid")
    for b in (B, 1, 3):
        ora.quantize_state()
        for l in range(3):
            h.set_weights(l, ora.w[l], ora.bias[l])
        x0, y = vectors(rng, b, n), vectors(rng, b, n)
        loss = h.train_step(torch.from_numpy(x0).cuda(), torch.from_numpy(y).cuda(), b, 0.1, want_loss=True)
        want = ora.train_step(x0, y, 0.1, keep=())["loss"]
        assert abs(loss - want) <= 1e-4 * want
        for l in range(3):
            check_close(h.get_weights(l, want_bias=False), ora.w[l], f"W^{l + 1} at B = {b}")
    h.destroy()


@pytest.mark.parametrize("sizes,kmax,cnt", [([1025, 15, 17, 1], 9, 33), ([16, 16, 16], 17, 64), ([1536, 2048 - 1536], 40, 96), ([128] * 12, 1, 32)])
def test_windowed_rows_sixteen_to_a_warp(torch_cuda, sizes, kmax, cnt):  # noqa: F811
    """The shared-memory window kernel for chunks of 32 inputs: groups short of a slice, one row over, of one row, the widest
    window, rows of one chunk pair and of several, weights read back in the caller's order."""
    rng = np.random.default_rng(sum(sizes) + kmax)
    n, start = sum(sizes), 0
    rows = []
    for size in sizes:
        for i in range(size):
            m = int(rng.integers(1, min(kmax, size) + 1))
            rows.append(np.sort(start + rng.choice(size, size=m, replace=False)))
        start += size
    rp = np.zeros(n + 1, dtype=np.int32)
    rp[1:] = np.cumsum([len(r) for r in rows])
    layers = 2
    arrays = ([rp] * layers, [np.concatenate(rows).astype(np.int32)] * layers,
              [(rng.standard_normal(rp[-1]) * 0.6).astype(np.float32) for _ in range(layers)],
              [(rng.standard_normal(n) * 0.1).astype(np.float32) for _ in range(layers)])
    pkg = sdnn()
    flags = pkg.FLAG_REORDER | pkg.FLAG_SMEM_WINDOWS
    infer_parity(torch_cuda, arrays, vectors(rng, cnt, n), 128, expect_nonempty=True, flags=flags)
    h = pkg.Sdnn.create(*arrays, max_batch=128, flags=flags)
    for l in range(layers):
        w, bias = h.get_weights(l)
        assert np.array_equal(w, arrays[2][l]) and np.array_equal(bias, arrays[3][l])
    h.destroy()


@pytest.mark.parametrize("flags", ["", "NO_PDL", "IDX32"])
def test_graphs_for_tiles_of_one_padded_width(torch_cuda, flags):  # noqa: F811
    """A handle asked for batches of many sizes: graphs that gather for exactly their inputs, graphs of more inputs that serve fewer, one
    that replaces another, two lanes of two tiles.  The sigmoid's padding is not zero, so anything it reached would show."""
    torch, pkg = torch_cuda, sdnn()
    rng = np.random.default_rng(8)
    n = 530
    arrays = ragged_net(rng, n=n, layers=5, kmax=40, scale=0.3)
    h = pkg.Sdnn.create(*arrays, max_batch=128, activation=pkg.ACT_SIGMOID, flags=getattr(pkg, "FLAG_" + flags) if flags else 0)
    ora = OracleNet(*arrays, activation="sigmoid")
    x0 = vectors(rng, 256, n)
    want, x = ora.infer(x0), torch.from_numpy(x0).cuda()
    for cnt in (128, 65, 72, 100, 128, 65, 3, 17, 80, 104, 127, 73, 128, 9, 200, 250, 193, 66, 256, 4):
        y = torch.full((cnt, n), -1.0, device="cuda")
        h.infer_batch(x, cnt, y)
        check_close(y.cpu().numpy(), want[:cnt], f"{cnt} inputs")
    h.destroy()


@pytest.mark.parametrize("cnt", [17, 33, 70, 96, 100, 300])
def test_windowed_tiles_of_whole_chunks(torch_cuda, cnt):  # noqa: F811
    """Nets with all their operands in shared memory: tiles padded to the next 32 columns, on a handle that has seen a wider one, in
    the first call and in later ones."""
    torch, pkg = torch_cuda, sdnn()
    rng = np.random.default_rng(cnt)
    n, size, layers, k = 1536, 512, 5, 24
    rp = np.arange(n + 1, dtype=np.int32) * k
    cols = [np.concatenate([np.sort(i // size * size + rng.choice(size, size=k, replace=False)) for i in range(n)]).astype(np.int32) for _ in range(layers)]
    vals = [(rng.standard_normal(n * k) * (2.0 / k) ** 0.5).astype(np.float32) for _ in range(layers)]
    bias = [(rng.standard_normal(n) * 0.1).astype(np.float32) for _ in range(layers)]
    h = pkg.Sdnn.create([rp] * layers, cols, vals, bias, max_batch=300, flags=pkg.FLAG_REORDER | pkg.FLAG_SMEM_WINDOWS)
    assert h.windowed_layers() == layers
    ora = OracleNet([rp] * layers, cols, vals, bias)
    wide = torch.from_numpy(vectors(rng, 300, n) + 5.0).cuda()
    h.infer_batch(wide, 300, torch.zeros(300, n, device="cuda"))
    for _ in range(3):
        x0 = vectors(rng, cnt, n)
        y, c = torch.full((cnt, n), -1.0, device="cuda"), torch.zeros(cnt, dtype=torch.int32, device="cuda")
        h.infer_batch(torch.from_numpy(x0).cuda(), cnt, y, c)
        got = y.cpu().numpy()
        check_close(got, ora.infer(x0), "x^L")
        assert np.array_equal(c.cpu().numpy(), np.count_nonzero(got, axis=1))
    h.destroy()


@pytest.mark.parametrize("mode", sorted(BWD_MODES))
@pytest.mark.parametrize("batches", [(17, 24, 25, 32), (40, 37, 33, 64, 56), (100, 65, 121, 128)])
def test_lanes_of_nothing_but_padding(torch_cuda, batches, mode):  # noqa: F811
    """Batches that leave whole lanes of a padded tile row empty, one handle for all of them: growing ones, smaller ones that run
    in the graph of a larger one, full ones.  The sigmoid's padding is not zero, so anything it reached would show."""
    torch, pkg = torch_cuda, sdnn()
    rng = np.random.default_rng(batches[0])
    n = 530
    arrays = ragged_net(rng, n=n, layers=3, kmax=40, scale=0.3)
    h = pkg.Sdnn.create(*arrays, max_batch=max(batches), train=True, update_bias=True, activation=pkg.ACT_SIGMOID, flags=BWD_MODES[mode])
    ora = OracleNet(*arrays, update_bias=True, activation="sigmoid")
    for b in batches:
        ora.quantize_state()
        for l in range(3):
            h.set_weights(l, ora.w[l], ora.bias[l])
        x0, y = vectors(rng, b, n), vectors(rng, b, n)
        h.train_step(torch.from_numpy(x0).cuda(), torch.from_numpy(y).cuda(), b, 0.5)
        ora.train_step(x0, y, 0.5, keep=())
        for l in range(3):
            w, bias = h.get_weights(l)
            check_close(w, ora.w[l], f"W^{l + 1} at B = {b}")
            check_close(bias, ora.bias[l], f"b^{l + 1} at B = {b}")
    h.destroy()
    for cnt in batches:
        infer_parity(torch_cuda, arrays, vectors(rng, cnt, n), max(batches), expect_nonempty=True)


def rowwise(rp, cols, vals, bias, x, act):
    """A layer in float64, entry by entry, so that what an entry does not read does not matter; NaN clamps to 0 as on the device."""
    out = np.empty((len(x), len(rp) - 1))
    for i in range(len(rp) - 1):
        with np.errstate(invalid="ignore"):
            z = bias[i] + (vals[rp[i]:rp[i + 1]].astype(np.float64) * x[:, cols[rp[i]:rp[i + 1]]]).sum(axis=1)
        out[:, i] = 1.0 / (1.0 + np.exp(-z)) if act == "sigmoid" else np.where(np.isnan(z), 0.0, np.clip(z, 0.0, 32.0))
    return out


@pytest.mark.parametrize("n,cnt,ragged", [(640, 1500, False), (1000, 590, True), (1024, 2400, False), (1025, 7105, True), (2047, 591, False), (2048, 1777, True), (2500, 900, True),
                                          (2700, 3000, False), (3585, 2368, True), (4096, 1777, False), (4608, 1184, False), (7200, 591, True), (8192, 592, False)])
def test_networks_held_in_shared_memory(torch_cuda, n, cnt, ragged):  # noqa: F811
    """Batches that go through whole networks in one launch (or two, for a last round of another width): 4 to 16 inputs a CTA, outputs
    that fit beside the inputs and outputs that wait in registers, last units and groups of eight of a few rows, empty rows, rows of 56; outputs
    and counts, ids, host buffers, and new weights."""
    torch, pkg = torch_cuda, sdnn()
    rng = np.random.default_rng(n)
    layers, act = 3, "clamped_relu" if n % 2 else "sigmoid"
    if ragged:
        rps, cols = [], []
        for _ in range(layers):
            length = rng.integers(0, 57, size=n)
            rps.append(np.concatenate([[0], np.cumsum(length)]).astype(np.int32))
            cols.append(np.concatenate([np.sort(rng.choice(n, size=m, replace=False)) for m in length]).astype(np.int32))
    else:
        rps, cols, _, _ = uniform_net(rng, n, 32, layers)
    vals = [(rng.standard_normal(len(c)) * 0.25).astype(np.float32) for c in cols]
    bias = [(rng.standard_normal(n) * 0.1).astype(np.float32) for _ in range(layers)]
    h = pkg.Sdnn.create(rps, cols, vals, bias, max_batch=min(cnt, 1024), activation=pkg.ACT_SIGMOID if act == "sigmoid" else pkg.ACT_CLAMPED_RELU)
    ora = OracleNet(rps, cols, vals, bias, activation=act)
    x0 = vectors(rng, cnt, n)
    x = torch.from_numpy(x0).cuda()
    pick = np.unique(np.concatenate([[0, cnt - 1], rng.integers(0, cnt, size=30)]))

    def call(**kw):
        y, c = torch.full((cnt, n), -1.0, device="cuda"), torch.full((cnt,), -1, dtype=torch.int32, device="cuda")
        before = h.kernel_launches()
        total = h.infer_batch(x, cnt, y, c, **kw)
        torch.cuda.synchronize()
        return y.cpu().numpy(), c.cpu().numpy(), total, h.kernel_launches() - before
    y, c, _, launches = call()
    assert launches <= 2, "one launch for whole rounds of CTAs, one for what is left"
    check_close(y[pick], ora.infer(x0[pick]), "x^L")
    assert np.array_equal(c, np.count_nonzero(y, axis=1))

    ids = torch.full((cnt * n,), -1, dtype=torch.int32, device="cuda")
    y2, c2, total, _ = call(nz_index_out=ids, nz_index_capacity=cnt * n, want_total=True)
    assert np.array_equal(y, y2) and np.array_equal(c, c2) and total == c.sum()
    ids = ids.cpu().numpy()
    assert np.array_equal(ids[:total], np.nonzero(y)[1]) and (ids[total:] == -1).all()

    ids2, c2 = torch.full((cnt * n,), -1, dtype=torch.int32, device="cuda"), torch.full((cnt,), -1, dtype=torch.int32, device="cuda")
    h.infer_batch(x, cnt, None, c2)                                # without the outputs: the same counts and ids
    assert np.array_equal(c2.cpu().numpy(), c)
    assert h.infer_batch(x, cnt, None, None, ids2, cnt * n, want_total=True) == total and np.array_equal(ids2.cpu().numpy(), ids)

    yh = np.empty((cnt, n), dtype=np.float32)
    h.infer_batch(x0, cnt, yh, None, host=True)
    check_close(yh[pick], ora.infer(x0[pick]), "x^L through host buffers")
    for l in range(layers):
        w, b = h.get_weights(l)
        assert np.array_equal(w, vals[l]) and np.array_equal(b, bias[l])

    vals = [(rng.standard_normal(len(c)) * 0.25).astype(np.float32) for c in cols]
    bias = [(rng.standard_normal(n) * 0.1).astype(np.float32) for _ in range(layers)]
    for l in range(layers):
        h.set_weights(l, vals[l], bias[l])
    y, c, _, _ = call()
    check_close(y[pick], OracleNet(rps, cols, vals, bias, activation=act).infer(x0[pick]), "x^L with new weights")

    # what no entry reads does not reach a row: infinities and NaN in some inputs' neurons
    x0[pick[1], :8] = np.inf
    x0[pick[2], n // 2] = np.nan
    x0[pick[3], n - 9:] = -np.inf
    x = torch.from_numpy(x0).cuda()
    y, c, _, _ = call()
    want = x0[pick[:5]].astype(np.float64)
    for l in range(layers):
        want = rowwise(rps[l], cols[l], vals[l], bias[l], want, act)
    assert np.array_equal(np.isnan(y[pick[:5]]), np.isnan(want))
    check_close(np.nan_to_num(y[pick[:5]]), np.nan_to_num(want), "x^L of inputs that are not finite")
    h.destroy()


@pytest.mark.parametrize("n,cnt,tile", [(640, 2000, 1024), (1024, 1000, 1000), (2048, 1500, 600), (4096, 2500, 1024), (4096, 592, 592),
                                        (1465, 449, 449), (1465, 200, 600), (700, 60, 100), (1500, 120, 128), (2000, 7, 40), (900, 1030, 1000)])
def test_dead_inputs_dropped_from_networks_held_in_shared_memory(torch_cuda, n, cnt, tile):  # noqa: F811
    """Inputs that die at once, after some layers, or not at all, dropped that way or, fewer of them, by the layer launches: the same bits as without dropping them, and the live inputs of the last tile
    after each layer; all inputs dead; none."""
    torch, pkg = torch_cuda, sdnn()
    rng = np.random.default_rng(n + cnt)
    layers, k = 14, 32
    rp, cols, _, _ = uniform_net(rng, n, k, layers)
    vals = [np.full(n * k, 1.0 / 16.0, dtype=np.float32)] * layers
    bias = [np.full(n, -0.35, dtype=np.float32)] * layers
    dense, drop = (pkg.Sdnn.create(rp, cols, vals, bias, max_batch=tile, flags=f) for f in (0, pkg.FLAG_SKIP_DEAD))
    mixed = (rng.random((cnt, n)) < rng.uniform(0.05, 0.5, size=(cnt, 1))).astype(np.float32)
    for x0 in (mixed, np.zeros_like(mixed), np.ones_like(mixed)):
        x, outs = torch.from_numpy(x0).cuda(), []
        for h in (dense, drop):
            y, c = torch.full((cnt, n), -1.0, device="cuda"), torch.full((cnt,), -1, dtype=torch.int32, device="cuda")
            ids = torch.full((cnt * n,), -1, dtype=torch.int32, device="cuda")
            total = h.infer_batch(x, cnt, y, c, ids, cnt * n, want_total=True)
            torch.cuda.synchronize()
            outs.append((y.cpu().numpy(), c.cpu().numpy(), ids.cpu().numpy(), total))
            live = list(h.get_liveness()) if h is drop else None
            c2, ids2 = torch.full_like(c, -1), torch.full_like(ids, -1)
            assert h.infer_batch(x, cnt, None, c2, ids2, cnt * n, want_total=True) == total      # the same without the outputs
            assert torch.equal(c, c2) and torch.equal(ids, ids2) and (live is None or list(h.get_liveness()) == live)
        assert all(np.array_equal(a, b) for a, b in zip(*outs))
        last = (cnt - 1) // drop.infer_tile_width() * drop.infer_tile_width()
        live, want = x0[last:], []
        for l in range(layers):
            live = np.clip(live[:, cols[l].reshape(n, k)].sum(axis=2) / 16.0 - 0.35, 0.0, 32.0)      # multiples of 1/16 from the 0/1 inputs of the first layer on
            want.append(int(live.any(axis=1).sum()))
            assert abs(int(drop.get_liveness()[l]) - want[-1]) <= 1, l      # rounding may keep the last neuron of an input alive
    dense.destroy()
    drop.destroy()


@pytest.mark.parametrize("n,B", [(17, 8), (700, 6), (700, 100), (1500, 33), (3001, 16), (6007, 37), (9000, 20)])
@pytest.mark.parametrize("ragged", [False, True])
def test_layers_that_do_not_fill_the_device(torch_cuda, n, B, ragged):  # noqa: F811
    """Train steps whose long rows and columns are split between groups of lanes (two, four, all of a warp's), trained and frozen biases."""
    rng = np.random.default_rng(n + B)
    if ragged:
        arrays = ragged_net(rng, n=n, layers=3, kmax=min(n, 60), scale=0.3)
    else:
        arrays = uniform_net(rng, n, min(n // 2, 32), 3)
    data = [(vectors(rng, B, n), vectors(rng, B, n)) for _ in range(2)]
    train_parity(torch_cuda, arrays, data, eta=0.02, update_bias=True, activation="sigmoid", expect_live=True)
    train_parity(torch_cuda, arrays, data[:1], eta=0.02, expect_live=True)


@pytest.mark.parametrize("n,cnt", [(5120, 3), (5121, 4), (5000, 7), (6001, 5), (4096, 12), (8192, 16), (8193, 9), (2048, 28), (4097, 20), (8000, 32), (17001, 28),
                                   (2048, 50), (4001, 64), (4097, 33), (2048, 100), (2049, 100), (1500, 250)])
def test_allocation_free_call_with_rows_shared_by_groups_of_lanes(torch_cuda, n, cnt):  # noqa: F811
    """One, two, four and eight groups of lanes to a row of the caller's CSR arrays, on either side of each rule; rows of 0 to 150 entries
    from any alignment, so that some take several steps of all groups and some not one."""
    torch, pkg = torch_cuda, sdnn()
    rng = np.random.default_rng(n + cnt)
    rp, cols, vals, bias = ragged_net(rng, n=n, layers=2, kmax=40, scale=0.3)
    for l in range(2):                                       # some rows much longer than the others
        length = np.diff(rp[l])
        length[rng.integers(0, n, size=20)] = 150
        rp[l] = np.concatenate([[0], np.cumsum(length)]).astype(np.int32)
        cols[l] = np.concatenate([np.sort(rng.choice(n, size=m, replace=False)) for m in length]).astype(np.int32)
        vals[l] = (rng.standard_normal(rp[l][-1]) * 0.3).astype(np.float32)
    at = [0, (len(cols[0]) + 3) // 4 * 4]
    col, val = np.zeros(at[1] + len(cols[1]), dtype=np.int32), np.zeros(at[1] + len(cols[1]), dtype=np.float32)
    for l in range(2):
        col[at[l]:at[l] + len(cols[l])] = cols[l]
        val[at[l]:at[l] + len(vals[l])] = vals[l]
    x0 = vectors(rng, cnt, n)
    got = torch.full((cnt, n), -1.0, device="cuda")
    pkg.infer_noalloc(2, n, *(torch.from_numpy(a).cuda() for a in (np.stack(rp), col, val)), np.asarray(at, dtype=np.int64),
                      torch.from_numpy(np.stack(bias)).cuda(), torch.from_numpy(x0).cuda(), cnt, got)
    torch.cuda.synchronize()
    check_close(got.cpu().numpy(), OracleNet(rp, cols, vals, bias).infer(x0), f"{n} neurons, {cnt} inputs")


@pytest.mark.parametrize("n,cnt", [(17, 8), (700, 6), (700, 100), (1500, 33), (3001, 16), (6007, 40), (9000, 20), (16000, 5), (17000, 64)])
@pytest.mark.parametrize("ragged", [False, True])
def test_inference_with_rows_shared_by_groups_of_lanes(torch_cuda, n, cnt, ragged):  # noqa: F811
    """Small batches through layers that do not fill the device, from the first call's launches and the later ones' graph, in a handle for just
    as many inputs and in one for more, with either index width."""
    torch, pkg = torch_cuda, sdnn()
    rng = np.random.default_rng(n + cnt)
    arrays = ragged_net(rng, n=n, layers=5, kmax=min(n, 60), scale=0.3) if ragged else uniform_net(rng, n, min(n // 2, 32), 5)
    x0 = vectors(rng, cnt, n)
    want, outs = OracleNet(*arrays).infer(x0), []
    for batch, flags in ((cnt, 0), (300, 0), (cnt, pkg.FLAG_IDX32)):
        h = pkg.Sdnn.create(*arrays, max_batch=batch, flags=flags)
        for _ in range(3):
            outs.append(torch.full((cnt, n), -1.0, device="cuda"))
            h.infer_batch(torch.from_numpy(x0).cuda(), cnt, outs[-1])
        torch.cuda.synchronize()
        h.destroy()
    check_close(outs[0].cpu().numpy(), want, "x^L")
    assert all(torch.equal(y, outs[0]) for y in outs)


@pytest.mark.parametrize("n,tile,cnt,host", [
    (1024, 1024, 1100, True), (2000, 600, 1250, True), (1500, 450, 455, True),      # whole networks in shared memory, a last tile too small for them
    (700, 100, 103, False), (700, 100, 106, True), (3000, 12, 29, False), (1500, 28, 60, False), (700, 8, 9, False),      # rows shared by groups of lanes
    (700, 300, 303, False), (4100, 400, 450, False), (4100, 257, 300, True), (700, 4, 11, False), (900, 256, 257, True)])
@pytest.mark.parametrize("kind", ["uniform", "ragged", "dying", "windows"])
def test_bits_do_not_depend_on_an_inputs_place_in_the_call(torch_cuda, n, tile, cnt, host, kind):  # noqa: F811
    """A call adds every input's sums in one order: the inputs of its last, narrower tile (or second half) are also its first ones, and give
    the same bits there; from the first call's launches and the later ones' graphs."""
    torch, pkg = torch_cuda, sdnn()
    rng = np.random.default_rng(n + cnt)
    layers, flags = 5, 0
    arrays = ragged_net(rng, n=n, layers=layers, kmax=60, scale=0.3) if kind == "ragged" else uniform_net(rng, n, 32, layers)
    if kind == "dying":
        flags = pkg.FLAG_SKIP_DEAD
        arrays = [*arrays[:2], [np.full(n * 32, 1.0 / 16.0, dtype=np.float32)] * layers, [np.full(n, -0.35, dtype=np.float32)] * layers]
    elif kind == "windows":
        flags = pkg.FLAG_REORDER | pkg.FLAG_SMEM_WINDOWS
        first = np.minimum(np.arange(n) // 100, n // 100 - 1) * 100      # blocks of 100 neurons, what is left belongs to the last one
        size = np.where(first == first[-1], n - first, 100)
        cols = [np.concatenate([np.sort(f + rng.choice(m, size=16, replace=False)) for f, m in zip(first, size)]).astype(np.int32) for _ in range(layers)]
        arrays = ([np.arange(n + 1, dtype=np.int32) * 16] * layers, cols, [rng.uniform(-1, 1, size=n * 16).astype(np.float32) for _ in range(layers)], arrays[3])
    h = pkg.Sdnn.create(*arrays, max_batch=tile, flags=flags)
    assert kind != "windows" or h.windowed_layers() == layers
    whole = min(tile, h.infer_tile_width())
    again = cnt % whole if cnt > tile else cnt // 3               # inputs that come twice
    x0 = vectors(rng, cnt, n) if kind != "dying" else (rng.random((cnt, n)) < rng.uniform(0.05, 0.5, size=(cnt, 1))).astype(np.float32)
    x0[cnt - again:] = x0[:again]
    for _ in range(3):
        if host:
            y = np.full((cnt, n), -1.0, dtype=np.float32)
            h.infer_batch(x0, cnt, y, host=True)
        else:
            yd = torch.full((cnt, n), -1.0, device="cuda")
            h.infer_batch(torch.from_numpy(x0).cuda(), cnt, yd)
            y = yd.cpu().numpy()
        assert np.array_equal(y[cnt - again:], y[:again])
    pick = np.unique(np.concatenate([[0, cnt - 1], rng.integers(0, cnt, size=10)]))
    if kind != "dying":
        check_close(y[pick], OracleNet(*arrays).infer(x0[pick]), "x^L")
    h.destroy()


def launched(torch, call, name):
    """Blocks of every launch that `call` makes of kernels of that name."""
    import json
    import os
    import tempfile
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA]) as p:
        call()
        torch.cuda.synchronize()
    with tempfile.TemporaryDirectory() as d:
        trace = os.path.join(d, "trace.json")
        p.export_chrome_trace(trace)
        with open(trace) as f:
            events = [e for e in json.load(f)["traceEvents"] if e.get("cat") == "kernel"]
    if not events:
        pytest.skip("no kernels in the trace")
    return [e["args"]["grid"][0] for e in events if name in e["name"]]


@pytest.mark.parametrize("n,k,B", [(3000, 64, 37), (6007, 32, 37), (2600, 112, 20)])
def test_column_units_leave_room_for_row_units_where_no_maps_are_made(torch_cuda, all_but, n, k, B):  # noqa: F811
    """A layer large enough for maps has none where the gradient is kept or memory does not allow it.  Its column units then run beside row
    units, and both fit the device (16 warps an SM) in one round; with maps the column units have it to themselves."""
    torch, pkg = torch_cuda, sdnn()
    rng = np.random.default_rng(n)
    arrays = uniform_net(rng, n, k, 3)
    x, y = (torch.from_numpy(vectors(rng, B, n)).cuda() for _ in range(2))
    slots = 16 * torch.cuda.get_device_properties(0).multi_processor_count
    groups = 32 // (8 if B > 32 else 4)
    rows, taken, weights = (n + groups - 1) // groups, [], []
    for flags in (0, pkg.FLAG_KEEP_DEBUG, 0):
        if len(taken) == 2:
            all_but(taken[0] + (40 << 20))                        # room for the net, not for what the maps leave to later calls
        h = pkg.Sdnn.create(*arrays, max_batch=B, train=True, activation=pkg.ACT_SIGMOID, flags=flags | pkg.FLAG_NO_GRAPH)
        taken.append(h.device_bytes())
        moves = launched(torch, lambda: h.train_step(x, y, B, 0.5), "split_values_kernel")
        units = launched(torch, lambda: h.train_step(x, y, B, 0.5), "backward_split_kernel")
        assert len(moves) == (2 if len(taken) == 1 else 0)
        assert all(u <= (slots if moves else slots - rows) for u in units) and (units or not moves)
        weights.append([h.get_weights(l, want_bias=False) for l in range(3)])
        h.destroy()
    for w in weights[1:]:
        for a, b in zip(w, weights[0]):
            check_close(a, b, "W after two steps")


@pytest.mark.parametrize("n,tile,cnt,quarter", [(4096, 640, 5000, False), (2048, 600, 3000, False), (2048, 1024, 3000, True)])
def test_nets_are_laid_out_twice_only_for_batches_of_the_handles_own_size(torch_cuda, all_but, n, tile, cnt, quarter):  # noqa: F811
    """A handle whose batches of max_batch inputs go through the layer launches holds its net once, whatever larger ones would take; and so does
    every handle made when less than a quarter of the device is free.  Larger batches give the same outputs."""
    torch, pkg = torch_cuda, sdnn()
    rng = np.random.default_rng(n)
    layers, k = 60, 32
    arrays = uniform_net(rng, n, k, layers)
    if quarter:
        all_but(torch.cuda.get_device_properties(0).total_memory // 5)
    h = pkg.Sdnn.create(*arrays, max_batch=tile, activation=pkg.ACT_SIGMOID)
    once = 6 * n * k * layers + 2 * 4 * n * ((tile + 255) // 256 * 256) + (24 << 20)      # entries, two tiles, lists and the last block of small arrays
    assert h.device_bytes() < once, (h.device_bytes(), once)
    x0 = vectors(rng, cnt, n)
    y = torch.full((cnt, n), -1.0, device="cuda")
    before = h.kernel_launches()
    h.infer_batch(torch.from_numpy(x0).cuda(), cnt, y)
    assert h.kernel_launches() - before > layers
    check_close(y[-8:].cpu().numpy(), OracleNet(*arrays, activation="sigmoid").infer(x0[-8:]), "x^L")
    h.destroy()


@pytest.mark.parametrize("n,cnt,drop", [(20011, 700, False), (20011, 900, True), (40000, 500, False), (40000, 400, True)])
def test_host_batches_of_wide_nets_keep_to_the_tile_width(torch_cuda, n, cnt, drop):  # noqa: F811
    """A batch within max_batch whose tiles are narrower for L2's sake goes in as many tiles from host memory as from device memory: the same launches, outputs,
    ids and live inputs of the last tile."""
    torch, pkg = torch_cuda, sdnn()
    rng = np.random.default_rng(n + cnt)
    layers, k = 3, 8
    arrays = uniform_net(rng, n, k, layers)
    if drop:
        arrays = [*arrays[:2], [np.full(n * k, 1.0 / 4.0, dtype=np.float32)] * layers, [np.full(n, -0.6, dtype=np.float32)] * layers]
    x0 = (rng.random((cnt, n)) < rng.uniform(0.0, 0.5, size=(cnt, 1)) ** 3).astype(np.float32) if drop else vectors(rng, cnt, n)
    x0[-3:] = 0.0
    h = pkg.Sdnn.create(*arrays, max_batch=cnt, flags=pkg.FLAG_SKIP_DEAD if drop else 0)
    T = h.infer_tile_width()
    assert T < cnt / 2
    outs = []
    for host in (False, True):
        y, c, ids = np.full((cnt, n), -1.0, dtype=np.float32), np.full(cnt, -1, dtype=np.int32), np.full(cnt * n, -1, dtype=np.int32)
        at = [torch.from_numpy(a) if host else torch.from_numpy(a).cuda() for a in (x0, y, c, ids)]
        args = [a.numpy() for a in at] if host else at
        before = h.kernel_launches()
        total = h.infer_batch(args[0], cnt, args[1], args[2], args[3], cnt * n, want_total=True, host=host)
        torch.cuda.synchronize()
        outs.append([a.cpu().numpy() for a in at[1:]] + [total, h.kernel_launches() - before, list(h.get_liveness()) if drop else None])
    assert all(np.array_equal(a, b) for a, b in zip(outs[0][:3], outs[1][:3])) and outs[0][3:] == outs[1][3:]
    if drop:
        last = (cnt - 1) // T * T
        assert outs[0][5][-1] == np.count_nonzero(outs[0][1][last:]) and 0 < outs[0][5][0] <= cnt - last
    pick = np.array([0, T, cnt - 1])
    check_close(outs[1][0][pick], OracleNet(*arrays).infer(x0[pick]), "x^L")
    h.destroy()


@pytest.mark.parametrize("n,cnt", [(500, 4100), (300, 8300), (700, 4160), (2048, 60), (1465, 100), (3000, 30), (9000, 33)])
def test_marks_of_live_inputs(torch_cuda, n, cnt):  # noqa: F811
    """Which inputs are alive after each layer, from launches whose marks meet per CTA and from smaller ones, and in batches of more columns than
    a CTA keeps marks for: the same bits as without dropping, and as many live inputs as have an output that is not zero."""
    torch, pkg = torch_cuda, sdnn()
    rng = np.random.default_rng(n + cnt)
    layers, k = 3, 256                                     # rows too long for whole networks in shared memory
    rp, cols, _, _ = uniform_net(rng, n, k, layers)
    vals, bias = [np.full(n * k, 1.0 / 128.0, dtype=np.float32)] * layers, [np.full(n, -0.35, dtype=np.float32)] * layers
    x0 = (rng.random((cnt, n)) < rng.uniform(0.0, 0.5, size=(cnt, 1))).astype(np.float32)
    x0[rng.random(cnt) < 0.3] = 0.0
    x, outs = torch.from_numpy(x0).cuda(), []
    for depth, flags in ((1, pkg.FLAG_SKIP_DEAD), (2, pkg.FLAG_SKIP_DEAD), (layers, pkg.FLAG_SKIP_DEAD), (layers, 0)):
        h = pkg.Sdnn.create(rp[:depth], cols[:depth], vals[:depth], bias[:depth], max_batch=cnt, flags=flags)
        assert h.infer_tile_width() == cnt
        y = torch.full((cnt, n), -1.0, device="cuda")
        h.infer_batch(x, cnt, y)
        outs.append(y.cpu().numpy())
        if flags:
            live = list(h.get_liveness())
            assert live == [np.count_nonzero(o.any(axis=1)) for o in outs] and 0 < live[0] < cnt
        h.destroy()
    assert np.array_equal(outs[2], outs[3])


@pytest.mark.parametrize("n,tile,cnt", [(1024, 1000, 3500), (2000, 592, 590), (1500, 450, 455)])
def test_counts_alone_take_no_running_total(torch_cuda, n, tile, cnt):  # noqa: F811
    """Host batches through whole networks in shared memory: the counts come with the outputs' launches; only a total or ids need more."""
    rng, pkg = np.random.default_rng(n), sdnn()
    arrays = uniform_net(rng, n, 32, 4)
    h = pkg.Sdnn.create(*arrays, max_batch=tile)
    x0 = vectors(rng, cnt, n)
    y, c, launches = np.empty((cnt, n), dtype=np.float32), np.full((2, cnt), -1, dtype=np.int32), []
    for args in ((y,), (y, c[0]), (None, c[1])):
        before = h.kernel_launches()
        h.infer_batch(x0, cnt, *args, host=True)
        launches.append(h.kernel_launches() - before)
    assert launches[0] == launches[1] == launches[2] < 4 * ((cnt + tile - 1) // tile), launches
    assert np.array_equal(c[0], np.count_nonzero(y, axis=1)) and np.array_equal(c[1], c[0])
    before = h.kernel_launches()
    assert h.infer_batch(x0, cnt, None, c[1], want_total=True, host=True) == c[0].sum() and h.kernel_launches() - before > launches[0]
    h.destroy()


@pytest.mark.parametrize("n,cnt,launches", [(4096, 592, True), (3001, 590, True), (1024, 1000, False), (1465, 449, False)])
def test_dead_inputs_dropped_after_new_weights(torch_cuda, n, cnt, launches):  # noqa: F811
    """Rows of several lengths with weights all different, so that an entry in another's place shows: the same bits with dead inputs dropped as without, through whole
    networks and through layer launches that stand in for them, from the first weights, from new ones, and from biases that end the dropping and
    begin it again."""
    torch, pkg = torch_cuda, sdnn()
    rng = np.random.default_rng(n + cnt)
    layers = 6
    rps, cols = [], []
    for _ in range(layers):
        length = rng.integers(8, 57, size=n)
        rps.append(np.concatenate([[0], np.cumsum(length)]).astype(np.int32))
        cols.append(np.concatenate([np.sort(rng.choice(n, size=m, replace=False)) for m in length]).astype(np.int32))

    def weights():
        return ([(rng.standard_normal(len(c)) * 0.22).astype(np.float32) for c in cols], [-rng.uniform(0.1, 0.3, size=n).astype(np.float32) for _ in range(layers)])
    vals, bias = weights()
    dense, drop = (pkg.Sdnn.create(rps, cols, vals, bias, max_batch=cnt, flags=f) for f in (0, pkg.FLAG_SKIP_DEAD))
    x0 = ((rng.random((cnt, n)) < 0.3) * np.exp(rng.uniform(np.log(0.02), np.log(20.0), size=(cnt, 1)))).astype(np.float32)
    x = torch.from_numpy(x0).cuda()

    def compare(dropping):
        outs, made = [], []
        for h in (dense, drop):
            y, c = torch.full((cnt, n), -1.0, device="cuda"), torch.full((cnt,), -1, dtype=torch.int32, device="cuda")
            before = h.kernel_launches()
            h.infer_batch(x, cnt, y, c)
            torch.cuda.synchronize()
            made.append(h.kernel_launches() - before)
            outs.append((y.cpu().numpy(), c.cpu().numpy()))
        assert all(np.array_equal(a, b) for a, b in zip(*outs))
        assert made[0] <= 2 and (made[1] > 2 * layers) == (launches and dropping), made
        if dropping:
            live = list(drop.get_liveness())
            assert live[-1] == np.count_nonzero(outs[1][1]) and 0 < live[-1] < live[0] < cnt, live
        pick = np.unique(np.concatenate([np.argsort(outs[0][1])[[0, cnt // 2, cnt - 1]], rng.integers(0, cnt, size=5)]))
        check_close(outs[1][0][pick], OracleNet(rps, cols, vals, bias).infer(x0[pick]), "x^L")
    compare(True)
    vals, bias = weights()
    for l in range(layers):
        for h in (dense, drop):
            h.set_weights(l, vals[l], bias[l])
    compare(True)
    kept, bias[2] = bias[2], bias[2].copy()
    bias[2][n // 2] = 0.25
    for h in (dense, drop):
        h.set_weights(2, None, bias[2])
    compare(False)
    bias[2], vals[4] = kept, weights()[0][4]
    for h in (dense, drop):
        h.set_weights(2, None, bias[2])
        h.set_weights(4, vals[4], None)
    compare(True)
    dense.destroy()
    drop.destroy()


@pytest.mark.parametrize("n,cnt,kmax", [(3000, 7, 16), (17000, 8, 40), (2000, 14, 30), (1500, 30, 24), (9201, 32, 24), (10999, 32, 60), (11001, 29, 60), (900, 50, 16), (700, 120, 14),
                                        (1701, 200, 60), (900, 300, 40), (1699, 256, 60), (5200, 4, 12)])
def test_allocation_free_call_with_short_rows(torch_cuda, n, cnt, kmax):  # noqa: F811
    """One group of lanes a row for short rows and on either side of the other lines, of lanes of 4 and of 8 inputs; layers with a gap behind them and
    a last one whose end the offsets do not tell."""
    torch, pkg = torch_cuda, sdnn()
    rng = np.random.default_rng(n + cnt)
    rp, cols, vals, bias = ragged_net(rng, n=n, layers=3, kmax=kmax, scale=0.3)
    at = [64]
    for c in cols[:-1]:
        at.append((at[-1] + len(c) + 3) // 4 * 4)
    at[2] += 128
    col, val = np.zeros(at[2] + len(cols[2]), dtype=np.int32), np.zeros(at[2] + len(cols[2]), dtype=np.float32)
    for l in range(3):
        col[at[l]:at[l] + len(cols[l])] = cols[l]
        val[at[l]:at[l] + len(vals[l])] = vals[l]
    x0 = vectors(rng, cnt, n)
    got = torch.full((cnt, n), -1.0, device="cuda")
    pkg.infer_noalloc(3, n, *(torch.from_numpy(a).cuda() for a in (np.stack(rp), col, val)), np.asarray(at, dtype=np.int64),
                      torch.from_numpy(np.stack(bias)).cuda(), torch.from_numpy(x0).cuda(), cnt, got)
    torch.cuda.synchronize()
    check_close(got.cpu().numpy(), OracleNet(rp, cols, vals, bias).infer(x0), f"{n} neurons, {cnt} inputs")
