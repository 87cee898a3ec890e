"""Data sketches of all modes from passes over A that serve two modes each (Alg. 1 part (a)): modes 0
and 1 from one read, the last one or two modes from another. Every mode against the oracle's sketch by
definition, in every storage type, at the edges of the passes' tiles: slabs of one and of several
chunks (10,240 entries; 5,120 in FP64), chunks that end inside a column, slabs on 16-, 8-, 4-, 2- and
1-byte boundaries, odd groups of tail indices, sketch sizes from fewer buckets than a CTA's threads
share up to 8192, more slabs than one CTA sorts, and tensors that start off the 16-byte grid. The
tolerance is the suite's for FP32 sums (1e-5 relative)."""
import threading

import numpy as np
import pytest

import tt_oracle as O
from paper_2309_08093_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2309_08093_gb300 import build as _build  # noqa: E402

_build.build()
from paper_2309_08093_gb300 import lib  # noqa: E402

TOL = 1e-5

SHAPES = [  # dims, J
    ((50, 50, 50), 1024),
    ((24, 23), 64),               # order 2: the head pass alone
    ((33, 31, 17), 512),          # odd columns
    ((101, 84, 9, 5), 128),       # eight lanes per bucket list
    ((128, 80, 3, 5), 2048),      # a slab of exactly 10,240 entries
    ((128, 81, 3, 5), 2047),      # one column more: two chunks; J not a power of two
    ((12, 11, 10, 9, 8), 4096),   # order 5: a mode between the passes
    ((6, 7, 29, 3, 2, 2), 1200),  # order 6: modes 0 and 1 without a pass
    ((30, 30, 14, 7, 3), 8192),   # several chunks, the largest J
    ((2048, 5, 6), 512),          # columns that leave four to a chunk
    ((8, 300, 5, 4), 45),
]


def _check(dims, J, dtype, offset=0, columns=None, rank=2):
    seed = 977
    a = synth.random_tensor(dims, 31)
    flat, scales, exact = synth.quantize(a, dtype)
    A = lib.device_tensor(np.concatenate([np.zeros(offset, flat.dtype), flat]), dtype)[offset:]
    sc = torch.from_numpy(scales).cuda() if scales is not None else None
    ctx = lib.Context(dims, [1] + [rank] * (len(dims) - 1) + [1], J, 1e-3, seed, dtype)
    Y = [torch.full((n, J), 3.0, device="cuda") for n in dims]
    for sweep in (4, 5):  # a second draw: accumulators and plans of the first are gone
        ctx.tt_sketch_unfold(A, -1, sweep, Y, sc)
    hs, vs = O.draw_sketch(seed, 5, dims, J)
    for k, n in enumerate(dims):
        cols = range(n) if columns is None else sorted({0, n // 2, n - 1})
        ref = np.stack([O.sketch_unfolding_column(exact, hs, vs, J, k, i) for i in cols])
        got = Y[k][list(cols)].double().cpu().numpy()
        err = np.linalg.norm(got - ref) / np.linalg.norm(ref)
        assert err <= TOL, (dims, J, dtype, k, err)
        # a bucket's error against the terms it sums: a lost or mis-signed term shows
        mag = np.stack([O.sketch_unfolding_column(np.abs(exact), hs, [np.ones_like(v) for v in vs], J, k, i)
                        for i in cols])
        assert np.all(np.abs(got - ref) <= TOL * (mag + np.abs(exact).max())), (dims, J, dtype, k)
    ctx.close()


@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16", "fp8"])
@pytest.mark.parametrize("dims,J", SHAPES)
def test_all_modes_against_the_oracle(dims, J, dtype):
    _check(dims, J, dtype)


@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16", "fp8"])
@pytest.mark.parametrize("dims,J", [
    ((1, 600, 5), 64), ((1, 32, 32, 8, 8), 256), ((1, 700, 3, 4), 512),  # first mode
    ((600, 1, 5), 64), ((32, 24, 1, 9), 256), ((24, 23, 1, 7, 5), 512),  # a middle one
    ((40, 30, 1), 64), ((32, 24, 9, 1), 256), ((1, 1, 600), 32), ((600, 1, 1, 1), 32),  # the last, several
])
def test_modes_of_size_one(dims, J, dtype):
    _check(dims, J, dtype, rank=1)


@pytest.mark.parametrize("dtype,offset", [("f32", 1), ("f32", 2), ("f64", 1), ("bf16", 1), ("bf16", 2), ("bf16", 4),
                                          ("fp8", 1), ("fp8", 2), ("fp8", 4), ("fp8", 8)])
def test_tensor_off_the_16_byte_grid(dtype, offset):
    _check((32, 24, 7, 5), 256, dtype, offset)


@pytest.mark.parametrize("n0", [6000, 14000, 24000, 40000])
def test_fp8_row_scales_beside_the_tail_chunk(n0):
    """A scale and a zero entry per row of A in shared memory: whole chunks, shorter ones, no tail pass."""
    _check((n0, 3, 4), 8192, "fp8", columns=3, rank=1)


@pytest.mark.parametrize("offset", [0, 4, 1])
def test_fp8_chunks_above_10240_entries(offset):
    """Four FP8 entries to a load reach 20,480 entries per chunk: slabs of two such chunks, and a base off
    the 4-byte grid, which goes one launch per mode."""
    _check((40, 30, 20, 5, 3), 2048, "fp8", offset, columns=3)


@pytest.mark.parametrize("row", [0, 13, 31])
def test_an_infinite_row_scale_stays_in_its_buckets(row):
    """FP8 with one infinite scale: a sum is not finite exactly where an entry of that row falls."""
    dims, J, seed = (32, 24, 7, 5), 4096, 977
    flat, scales, _ = synth.quantize(synth.random_tensor(dims, 31), "fp8")
    scales = scales.copy()
    scales[row] = np.inf
    ctx = lib.Context(dims, [1, 2, 2, 2, 1], J, 1e-3, seed, "fp8")
    Y = [torch.empty(n, J, device="cuda") for n in dims]
    ctx.tt_sketch_unfold(lib.device_tensor(flat, "fp8"), -1, 4, Y, torch.from_numpy(scales).cuda())
    hs, vs = O.draw_sketch(seed, 4, dims, J)
    hit = np.zeros(dims)
    hit[row] = 1.0
    ones = [np.ones_like(v) for v in vs]
    for k, n in enumerate(dims):
        bad = np.stack([O.sketch_unfolding_column(hit, hs, ones, J, k, i) for i in range(n)]) > 0
        assert np.array_equal(~np.isfinite(Y[k].cpu().numpy()), bad), k
    ctx.close()


@pytest.mark.parametrize("dims,J", [((32, 24, 7, 5), 4096), ((32, 24, 7, 5), 1024), ((23, 31, 6), 2048)])
def test_an_infinite_row_scale_keeps_its_sign(dims, J):
    """FP8 with one infinite scale: a bucket that one non-zero entry of that row falls into holds its signed
    infinity, whatever else it sums."""
    seed, row = 977, 13
    flat, scales, exact = synth.quantize(synth.random_tensor(dims, 31), "fp8")
    scales = scales.copy()
    scales[row] = np.inf
    ctx = lib.Context(dims, [1] + [2] * (len(dims) - 1) + [1], J, 1e-3, seed, "fp8")
    Y = [torch.empty(n, J, device="cuda") for n in dims]
    ctx.tt_sketch_unfold(lib.device_tensor(flat, "fp8"), -1, 4, Y, torch.from_numpy(scales).cuda())
    hs, vs = O.draw_sketch(seed, 4, dims, J)
    hit, value = np.zeros(dims), np.zeros(dims)
    hit[row] = 1.0
    value[row] = exact[row]
    ones = [np.ones_like(v) for v in vs]
    for k, n in enumerate(dims):
        one = np.stack([O.sketch_unfolding_column(hit, hs, ones, J, k, i) for i in range(n)]) == 1
        val = np.stack([O.sketch_unfolding_column(value, hs, vs, J, k, i) for i in range(n)])
        one &= val != 0
        assert one.any() and np.array_equal(Y[k].cpu().numpy()[one], np.copysign(np.inf, val[one])), k
    ctx.close()


@pytest.mark.parametrize("slabs", [40, 120, 240])
def test_accumulators_near_their_bound(slabs):
    """700 x 300 slabs at J = 8192: a head pass with the copies its sums ask for, with half of them, and none."""
    _check((700, 300, slabs), 8192, "f32", columns=3, rank=1)


def test_more_slabs_than_one_cta_sorts():
    """33,800 slabs of 512 entries: the head pass takes them from mode 1's grid-wide plan."""
    _check((32, 16, 130, 260), 1024, "f32", columns=3)


def test_a_workspace_cap_that_leaves_no_room_for_the_passes():
    """A cap between the needs of one launch per mode and of the passes: the context is created, and
    its sketches are the same."""
    dims, J, seed = (40, 36, 10, 9), 1024, 5
    ranks = (1, 2, 2, 2, 1)
    A = lib.device_tensor(synth.quantize(synth.random_tensor(dims, 3), "f32")[0], "f32")
    Y = [[torch.empty(n, J, device="cuda") for n in dims] for _ in range(2)]
    ctx = lib.Context(dims, ranks, J, 1e-3, seed)
    ctx.tt_sketch_unfold(A, -1, 0, Y[0])
    ctx.close()
    lo, hi = 1 << 16, 1 << 26  # smallest cap that still creates a context
    prev = lib.tt_set_workspace_limit(0)
    try:
        while hi - lo > 4096:
            mid = (lo + hi) // 2
            lib.tt_set_workspace_limit(mid)
            try:
                lib.Context(dims, ranks, J, 1e-3, seed).close()
                hi = mid
            except lib.TtError:
                lo = mid
        lib.tt_set_workspace_limit(hi)
        ctx = lib.Context(dims, ranks, J, 1e-3, seed)
    finally:
        lib.tt_set_workspace_limit(prev)
    ctx.tt_sketch_unfold(A, -1, 0, Y[1])
    for a, b in zip(*Y):
        assert float(torch.linalg.vector_norm(a - b)) <= TOL * float(torch.linalg.vector_norm(a))
    ctx.close()


def test_a_workspace_cap_leaves_room_for_the_host_calls():
    """The smallest cap under which one launch per mode and the host-buffer calls' staging fit: the passes'
    workspaces must not take that room."""
    dims, J, ranks = (40, 36, 30, 9), 64, (1, 2, 2, 2, 1)
    flat = synth.quantize(synth.random_tensor(dims, 3), "f32")[0]
    cores = [np.asarray(g, np.float32).ravel(order="F").copy() for g in synth.random_tt(dims, ranks, 4)]
    stage = 2 * (4 * flat.size + 4 * dims[0]) + sum(4 * g.size for g in cores)
    lo, hi = 1 << 16, 1 << 26  # smallest cap that still creates a context
    prev = lib.tt_set_workspace_limit(0)
    try:
        while hi - lo > 64:
            mid = (lo + hi) // 2
            lib.tt_set_workspace_limit(mid)
            try:
                lib.Context(dims, ranks, J, 1e-3, 5).close()
                hi = mid
            except lib.TtError:
                lo = mid
        lib.tt_set_workspace_limit(hi + stage)
        ctx = lib.Context(dims, ranks, J, 1e-3, 5)
        ctx.tt_prox_als_sweep_host(np.ascontiguousarray(flat, np.float32), cores, 1)
        ctx.close()
    finally:
        lib.tt_set_workspace_limit(prev)


def test_contexts_of_different_shapes_in_threads():
    """Contexts whose launches of one kernel need different amounts of shared memory, each driven by a thread
    of its own: every call succeeds, and the sketches are those of calls from one thread."""
    shapes = [((20, 30, 6, 5), 64), ((100, 100, 4, 3), 1024), ((40, 16, 6, 5), 128), ((100, 90, 4, 3), 1000)]
    work = []
    for dims, J in shapes:
        ctx = lib.Context(dims, (1, 2, 2, 2, 1), J, 1e-3, 5)
        A = lib.device_tensor(synth.quantize(synth.random_tensor(dims, 3), "f32")[0], "f32")
        Y = [[torch.empty(n, J, device="cuda") for n in dims] for _ in range(2)]
        ctx.tt_sketch_unfold(A, -1, 0, Y[0])
        work.append((ctx, A, Y))
    torch.cuda.synchronize()
    errors, start = [], threading.Barrier(len(work))

    def drive(ctx, A, Y):
        start.wait()
        try:
            for t in range(400):
                ctx.tt_sketch_unfold(A, -1, t % 2, Y[1])  # two draws in turn: plans too
                ctx.tt_sketch_unfold(A, t % 4, t % 2, Y[1])
            ctx.tt_sketch_unfold(A, -1, 0, Y[1])
        except lib.TtError as e:
            errors.append(e)

    threads = [threading.Thread(target=drive, args=w) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors[0]
    for ctx, _, Y in work:
        for a, b in zip(*Y):
            assert float(torch.linalg.vector_norm(a - b)) <= TOL * float(torch.linalg.vector_norm(a))
        ctx.close()


# Rounding of FP32 sums: n adds one after the other, each off by at most 2^-24 of the partial sum, leave a
# relative error of at most about 2^-24 sqrt(n / 2) of a sum of n terms of random sign (the partial sums
# grow with the square root); the levels of a sum (a bucket's entries of one slab, the slabs of one copy,
# the copies in pairs) add in squares.
def _chain_bound(*levels):
    return 2.0**-24 * np.sqrt(sum(n / 2 for n in levels))


@pytest.mark.parametrize("dims,J,dtype,k,levels", [
    ((64, 170, 2, 400), 512, "f32", 2, (11, 25, 10)),  # 800 slab chunks per bucket, 32 copies
    ((64, 170, 400, 2), 512, "f32", 3, (11, 25, 10)),  # its registers' runs cut, 8 copies
    ((40, 16, 90, 60), 64, "f32", 0, (2, 25, 1)),      # 3,100 runs of 16 columns: 775 adds, 32 copies
    ((40, 16, 90, 60), 64, "f32", 1, (2, 61, 1)),      # ... of 40 rows: 1,940 adds, 32 copies
    ((40, 16, 90, 60), 64, "fp8", 0, (2, 2, 1)),       # sums of unscaled FP8 entries are exact
])
def test_long_sums_keep_their_accuracy(dims, J, dtype, k, levels):
    """Few columns and many slabs: buckets that take hundreds of adds."""
    seed = 977
    flat, scales, exact = synth.quantize(synth.random_tensor(dims, 31), dtype)
    ctx = lib.Context(dims, [1, 2, 2, 2, 1], J, 1e-3, seed, dtype)
    Y = [torch.empty(n, J, device="cuda") for n in dims]
    sc = torch.from_numpy(scales).cuda() if scales is not None else None
    ctx.tt_sketch_unfold(lib.device_tensor(flat, dtype), -1, 5, Y, sc)
    hs, vs = O.draw_sketch(seed, 5, dims, J)
    ref = np.stack([O.sketch_unfolding_column(exact, hs, vs, J, k, i) for i in range(2)])
    err = np.linalg.norm(Y[k][:2].double().cpu().numpy() - ref) / np.linalg.norm(ref)
    assert err <= _chain_bound(*levels), err
    ctx.close()
