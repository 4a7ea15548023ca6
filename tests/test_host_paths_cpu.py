"""Host paths of the library on a stand-in CUDA runtime (host_only.py): what the entry points
allocate, launch and leave behind where a real device would have to fail or be probed."""

import ctypes

import numpy as np
import pytest

from tests.host_only import Library


@pytest.fixture()
def lib():
    lib = Library()
    yield lib
    lib.hook(None)
    lib.fake_fail_alloc(0)
    lib.fake_fail_copy(0)


def ints(address, n):
    return (ctypes.c_int32 * n).from_address(address)


def words(address, n):
    return [v or 0 for v in (ctypes.c_uint64 * n).from_address(address)]


@pytest.mark.parametrize("first", ["run", "tune", "load_state"])
@pytest.mark.parametrize("reload", [0, 1])
def test_a_search_that_ran_out_of_memory_leaves_nothing_behind(lib, first, reload):
    """Whichever allocation of a search fails, the call says EBIC_ENOMEM, and the same call (after a
    reload of the matrix or not) allocates anew: no launch gets the buffers that are missing."""
    ebic = lib.ebic
    p = ebic.Params.make(pop_size=100, max_len=6, init_max_len=6, elite=2, n_biclusters=3, mode=1)
    ci = np.tile(np.arange(2, dtype=np.int32), 10)
    off = np.arange(0, 22, 2, dtype=np.int32)
    null = []

    def check(kernel, grid, args):
        if "k_reset" in kernel:
            seg = words(args[0], 28)
            null.extend(k for k in range(14) if seg[14 + k] and not seg[k])
        if "k_init" in kernel:
            null.extend(k for k in range(8) if not words(args[1], 8)[k])

    before = lib.fake_device_blocks()
    lib.hook(check)
    blob = np.zeros(1 << 20, np.uint8)
    ctx = lib.context()
    assert lib.load(ctx, 300, 20) == 0
    assert lib.run(ctx, p, 1)[0] == 0
    size = lib.ebic_state_bytes(ctx)
    assert 0 < size <= blob.size and lib.ebic_save_state(ctx, blob.ctypes.data, size) == 0
    lib.ebic_destroy(ctx)

    def begin(ctx):
        if first == "run":
            return lib.run(ctx, p, 1)[0]
        if first == "load_state":
            return lib.ebic_load_state(ctx, ctypes.byref(p), blob.ctypes.data, size)
        return lib.ebic_autotune(ctx, ci.ctypes.data, off.ctypes.data, 10, ctypes.byref(p), 5, None)

    failed = 0
    for n in range(1, 200):
        ctx = lib.context()
        assert lib.load(ctx, 300, 20) == 0
        lib.fake_fail_alloc(n)
        st = begin(ctx)
        lib.fake_fail_alloc(0)
        if st == 0:
            lib.ebic_destroy(ctx)
            break
        assert st == ebic.EBIC_ENOMEM
        failed += 1
        if reload:
            assert lib.load(ctx, 300, 20) == 0
        assert lib.run(ctx, p, 1)[0] == 0
        lib.ebic_destroy(ctx)
    assert failed > 25 and n < 199
    assert not null
    assert lib.fake_device_blocks() == before


@pytest.mark.parametrize("at,written", [
    ((0, 1024, 2048, 4096), (1, 1, 1, 1)),            # apart, on their boundaries: all in place
    ((0, 1024, 2048, 4100), (0, 0, 0, 0)),            # fitness between two boundaries
    ((2, 1024, 2048, 4096), (0, 0, 0, 0)), ((0, 1024, 2049, 4096), (0, 0, 0, 0)),
    ((0, 0, 2048, 4096), (0, 0, 0, 0)),               # one over another
    ((0, 1024, 2048, 2176), (0, 0, 0, 0)),
    ((8192, 1024, 2048, 4096), (0, 0, 0, 0)),         # over the offsets
    ((8192 - 396, 1024, 2048, 4096), (0, 0, 0, 0)), ((8192 - 400, 1024, 2048, 4096), (1, 1, 1, 1)),
    ((None, 1024, None, 4100), (0, 0, 0, 0)), ((None, 1024, None, 4104), (0, 1, 0, 1))])
def test_device_outputs_are_written_in_place_only_where_they_can_be(lib, at, written):
    """100 individuals; outputs at byte offsets of one device block, the population's offsets at
    8,192.  What is not written in place is copied there, outputs in their order."""
    n = 100
    seen, copied = [], []

    def look(kernel, grid, args):
        if "k_sweep_finish" in kernel:
            seen.extend(words(args[3], 4))
            copied.append(lib.fake_calls(b"copy"))

    ctx = lib.context()
    assert lib.load(ctx, 300, 20) == 0
    block = lib.device(1 << 14)
    cols = lib.device(4 * 2 * n)
    off = np.arange(0, 2 * n + 2, 2, dtype=np.int32)
    ctypes.memmove(block + 8192, off.ctypes.data, off.nbytes)
    outs = [None if o is None else block + o for o in at]
    p = lib.ebic.Params.make(mode=1)
    lib.hook(look)
    lib.fake_clear_log()
    assert lib.ebic_eval_population(ctx, cols, block + 8192, n, ctypes.byref(p), *outs) == 0
    assert [int(s == o) for s, o in zip(seen, [o or 0 for o in outs])] == \
        [1 if o is None and k < 3 else w for k, (o, w) in enumerate(zip(outs, written))]
    assert all(s % (8 if k == 3 else 4) == 0 for k, s in enumerate(seen))
    wanted = sum(o is not None for o in outs)
    assert lib.fake_calls(b"copy") - copied[0] == wanted - sum(written)
    lib.ebic_destroy(ctx)


@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("device", [0, 1])
def test_a_refused_population_builds_nothing(lib, mode, device):
    """A population that the check refuses is refused before the form's bitmap or rank codes are
    built (there may be no memory for them), and the next good one is evaluated."""
    n = 800                       # (AUTO: the bitmap pays for device and host populations alike)
    ci = np.tile(np.arange(20, dtype=np.int32), n)
    off = np.arange(0, 20 * n + 20, 20, dtype=np.int32)
    bad = True

    def check(kernel, grid, args):     # what the first and the last launch write of the check
        if "k_sweep_prepare" in kernel:
            ints(words(args[5], 1)[0], 3)[1] = 2 * bad
            if words(args[8], 1)[0]:
                ends = ints(words(args[8], 1)[0], 3)
                ends[0], ends[1] = 0, 20 * n
                if bad:
                    ends[2] = 1
        if "k_sweep_finish" in kernel:
            ints(words(args[4], 1)[0], 1)[0] = ints(words(args[2], 1)[0], 3)[1]

    lib.hook(check)
    ctx = lib.context()
    assert lib.load(ctx, 3000, 20) == 0
    a, o = ci.ctypes.data, off.ctypes.data
    if device:
        a, o = lib.device(ci.nbytes), lib.device(off.nbytes)
        ctypes.memmove(a, ci.ctypes.data, ci.nbytes)
        ctypes.memmove(o, off.ctypes.data, off.nbytes)
    out = np.zeros(n, np.int32)
    p = lib.ebic.Params.make(mode=mode)

    def call():
        lib.fake_clear_log()
        st = lib.ebic_eval_population(ctx, a, o, n, ctypes.byref(p), out.ctypes.data, None, None, None)
        return st, [k for k, _ in lib.log()]

    st, ran = call()
    assert st == lib.ebic.EBIC_EINVAL
    assert len(ran) == 1 and "k_sweep_prepare" in ran[0]
    assert lib.ebic_copy_bitmap(ctx, out.ctypes.data, 1 << 30) == lib.ebic.EBIC_ESTATE
    bad = False
    st, ran = call()
    assert st == 0 and any("k_rank_codes" in k for k in ran) and "k_sweep_finish" in ran[-1]
    lib.ebic_destroy(ctx)


@pytest.mark.parametrize("call,copy", [("load", 2), ("evaluate", 3), ("tune", 3)])
def test_an_error_that_was_never_read_does_not_reach_the_next_load(lib, call, copy):
    """A load (NaN in the matrix) or a population check (a bad chromosome) whose result could not be
    read: the copy fails, and the next load of a good matrix is accepted."""
    bad = True

    def check(kernel, grid, args):
        if bad and "k_upload" in kernel and call == "load":
            ints(words(args[5], 1)[0], 1)[0] = 1
        if bad and "k_validate_csr" in kernel:
            ints(words(args[4], 1)[0], 1)[0] = 2

    lib.hook(check)
    ctx = lib.context()
    ci, off = np.zeros(8, np.int32), np.arange(0, 10, 2, dtype=np.int32)
    p = lib.ebic.Params.make(mode=3)                   # (the plain form)
    if call != "load":
        assert lib.load(ctx, 300, 20) == 0
    lib.fake_fail_copy(copy)
    if call == "load":
        assert lib.load(ctx, 300, 20) == lib.ebic.EBIC_ECUDA
    elif call == "evaluate":
        assert lib.ebic_eval_population(ctx, ci.ctypes.data, off.ctypes.data, 4, ctypes.byref(p),
                                        None, None, None, None) == lib.ebic.EBIC_ECUDA
    else:
        assert lib.ebic_autotune(ctx, ci.ctypes.data, off.ctypes.data, 4, ctypes.byref(p), 1,
                                 None) == lib.ebic.EBIC_ECUDA
    lib.fake_fail_copy(0)
    bad = False
    assert lib.load(ctx, 300, 20) == 0
    lib.ebic_destroy(ctx)


@pytest.mark.parametrize("graph", [0, 1])
@pytest.mark.parametrize("fuse,form", [(0, "k_evolve_block"), (-1, "k_evolve"), (2, "k_evolve")])
def test_the_counters_count_the_launches_made(lib, fuse, form, graph):
    """A search of 21 generations (a chunk of sixteen and singles in graph replays): the evaluation,
    evolve and scoring counters are the launches made, with no evaluation launch per generation
    where k_evolve_block evaluates; with statistics on (eager here) it does have one."""
    ebic = lib.ebic
    p = ebic.Params.make(pop_size=100, max_len=6, init_max_len=6, elite=2, n_biclusters=3, mode=2,
                         fuse_pairs=fuse, use_graph=graph, tabu_hit_limit=0)
    ctx = lib.context()
    assert lib.load(ctx, 300, 20) == 0

    def made(part):
        return sum(part in k for k, _ in lib.log())

    def counted(kernel):
        st = ebic.KernelStats()
        assert lib.ebic_profile_read(ctx, kernel, ctypes.byref(st)) == 0
        return st.launches

    for timed in (0, 1) if not graph else (0,):
        assert lib.ebic_profile_enable(ctx, 1) == 0
        assert lib.ebic_profile_enable(ctx, timed) == 0
        lib.fake_clear_log()
        st, rep = lib.run(ctx, p, 21)
        assert st == 0
        evals, evolves, ends = made("k_eval_bitmap"), made("k_evolve"), made("k_finish")
        first = 1 - timed                            # (the initial population, scored once)
        assert evolves == 21 and ends == 21 + first
        assert evals == first + (0 if form == "k_evolve_block" and not timed else 21)
        assert (made("k_evolve_block") > 0) == (form == "k_evolve_block" and not timed)
        assert counted(ebic.KERNEL_EVAL) == evals
        assert counted(ebic.KERNEL_EVOLVE) == evolves
        assert counted(ebic.KERNEL_FINISH) == ends
        assert counted(ebic.KERNEL_ALL) == len(lib.log())
    lib.ebic_destroy(ctx)


def test_tuned_sizes_are_for_matrices_of_the_same_kind_of_ties(lib):
    """Tuned on a matrix with few tied pairs (later candidates time faster here, so the tuner picks
    the last ones): a reload without many ties runs the same launches, one with many ties those
    of a context that was never tuned, and after it one with few again the tuned ones."""
    ebic = lib.ebic
    R, C = 4500, 650                                  # (243 MB of pair words: larger than L2)
    tied = 0

    def count(kernel, grid, args):
        if "k_count_tied" in kernel:
            ints(words(args[3], 1)[0], 1)[0] = tied

    lib.hook(count)
    ci = np.arange(600, dtype=np.int32)
    off = np.arange(0, 606, 6, dtype=np.int32)
    p = ebic.Params.make(pop_size=2000, max_len=6, init_max_len=6, elite=2, n_biclusters=3, mode=0,
                         tabu_hit_limit=0, neg_trends=1, ratio_num=85, ratio_den=100)

    def launches(ctx, n_tied):
        nonlocal tied
        tied = n_tied
        assert lib.load(ctx, R, C) == 0 and lib.ebic_build_bitmap(ctx) == 0
        lib.fake_clear_log()
        assert lib.ebic_eval_population(ctx, ci.ctypes.data, off.ctypes.data, 100, ctypes.byref(p),
                                        None, None, None, None) == 0
        st, rep = lib.run(ctx, p, 3)
        assert st == 0
        return [(k, g) for k, g in lib.log() if "k_eval" in k or "k_evolve" in k], rep.fuse_pairs

    many = C * C
    ctx, plain = lib.context(), lib.context()
    untuned = {n: launches(plain, n) for n in (0, many)}
    tied = 0
    assert lib.load(ctx, R, C) == 0 and lib.ebic_build_bitmap(ctx) == 0
    lib.fake_elapsed(1000.0, -0.01)
    rep = ebic.TuneReport()
    assert lib.ebic_autotune(ctx, ci.ctypes.data, off.ctypes.data, 100, ctypes.byref(p), 100,
                             ctypes.byref(rep)) == 0
    assert rep.mode == ebic.MODE_BITMAP and (rep.ipw_bitmap, rep.ipw_loop, rep.fuse_loop) == (4, 4, 63)
    tuned = launches(ctx, 0)
    assert tuned[1] == 63 and tuned != untuned[0]
    assert launches(ctx, many) == untuned[many]
    assert launches(ctx, 0) == tuned
    for c in (ctx, plain):
        lib.ebic_destroy(c)


@pytest.mark.parametrize("rows,cols", [(4225, 300), (40_000, 100), (5000, 1100)])
@pytest.mark.parametrize("call", ["evaluate", "tune"])
def test_auto_takes_the_bitmap_where_what_it_allocates_is_half_of_the_free_memory(lib, rows, cols, call):
    """AUTO and the autotuner weigh what the build really allocates (padded pair rows, bit planes,
    pair counts): with one byte of free memory less than twice that, there is no bitmap."""
    ebic = lib.ebic
    n = 16_000                                        # (enough sweeps' work for the cost model)
    ci = np.tile(np.arange(20, dtype=np.int32), n)
    off = np.arange(0, 20 * n + 20, 20, dtype=np.int32)
    p = ebic.Params.make(mode=0)

    def look(kernel, grid, args):                     # (the population is good; its ends)
        if "k_sweep_prepare" in kernel and words(args[8], 1)[0]:
            ints(words(args[8], 1)[0], 3)[1] = 20 * n

    lib.hook(look)

    def build_bytes():
        """What ebic_build_bitmap allocates over rank codes that are there already."""
        ctx = lib.context()
        q = ebic.Params.make(mode=1)
        assert lib.load(ctx, rows, cols) == 0
        assert lib.ebic_eval_population(ctx, ci.ctypes.data, off.ctypes.data, 1, ctypes.byref(q),
                                        None, None, None, None) == 0
        before = lib.fake_device_bytes()
        assert lib.ebic_build_bitmap(ctx) == 0
        got = lib.fake_device_bytes() - before
        lib.ebic_destroy(ctx)
        return got

    def takes_bitmap(free):
        lib.fake_set_free(free)
        ctx = lib.context()
        assert lib.load(ctx, rows, cols) == 0
        if call == "tune":
            assert lib.ebic_autotune(ctx, ci.ctypes.data, off.ctypes.data, n, ctypes.byref(p), 2,
                                     None) == 0
        else:
            assert lib.ebic_eval_population(ctx, ci.ctypes.data, off.ctypes.data, n,
                                            ctypes.byref(p), None, None, None, None) == 0
        lib.fake_clear_log()
        st = lib.ebic_copy_bitmap(ctx, None, 0)       # (EBIC_ESTATE: no bitmap)
        lib.ebic_destroy(ctx)
        return st != ebic.EBIC_ESTATE

    need = build_bytes()
    assert takes_bitmap(2 * need + 2)
    assert not takes_bitmap(2 * need - 2)


@pytest.mark.parametrize("rows,cols", [(300, 20), (10_000, 100), (33_333, 777), (5000, 1100)])
@pytest.mark.parametrize("mode", [1, 2])
def test_a_jobs_footprint_is_what_it_allocates(lib, rows, cols, mode):
    """The server reserves what a job's search allocates, and no more than its 1/16 slack and a few
    small buffers beyond it: a job of the direct form reserves nothing for the bitmap's planes."""
    p = lib.ebic.Params.make(pop_size=400, max_len=8, init_max_len=8, mode=mode, tabu_hit_limit=0)
    foot = lib.ebic_job_footprint(rows, cols, ctypes.byref(p), 20)
    before = lib.fake_device_bytes()
    ctx = lib.context()
    assert lib.load(ctx, rows, cols) == 0
    assert lib.run(ctx, p, 20)[0] == 0
    used = lib.fake_device_bytes() - before
    lib.ebic_destroy(ctx)
    assert used <= foot <= used * 17 / 16 + 16384


@pytest.mark.parametrize("rows,cols,device,packs,strided,plain", [
    (4225, 300, 1, 1, 0, 0), (33_333, 200, 1, 1, 0, 0), (33_333, 50, 0, 1, 0, 1),
    (4225, 300, 0, 2, 0, 2), (4225, 520, 0, 4, 0, 4), (33_333, 200, 0, 0, 1, 0),
    (4096, 300, 1, 0, 0, 1), (4096, 300, 0, 0, 0, 1)])
def test_padded_pair_rows_go_out_packed(lib, rows, cols, device, packs, strided, plain):
    """ebic_copy_bitmap: packed by a kernel for the device and, whole or in pieces, for the host where
    rows are short or the bitmap is small; unpadded rows as one copy."""
    ctx = lib.context()
    assert lib.load(ctx, rows, cols) == 0 and lib.ebic_build_bitmap(ctx) == 0
    n = lib.ebic_bitmap_bytes(rows, cols) // 4
    out = np.empty(n, np.uint32)
    dst = lib.device(4 * n) if device else out.ctypes.data
    lib.fake_clear_log()
    assert lib.ebic_copy_bitmap(ctx, dst, n) == 0
    assert sum("k_copy_rows" in k for k, _ in lib.log()) == packs
    assert (lib.fake_calls(b"copy2d"), lib.fake_calls(b"copy")) == (strided, plain)
    lib.ebic_destroy(ctx)


def test_contexts_are_made_of_kept_blocks(lib):
    """A context takes one device allocation; its pinned block goes back for the next one, up to as
    many as a job server has workers (64), and no further."""
    def several(n):
        lib.fake_fail_alloc(0)
        ctxs = [lib.context() for _ in range(n)]
        made = lib.fake_allocs()
        for c in ctxs:
            lib.ebic_destroy(c)
        return made

    before = lib.fake_device_blocks()
    several(64)
    kept = lib.fake_pinned_blocks()
    assert kept == 64
    assert several(64) == 64                          # (no pinned block anew)
    assert several(70) == 76
    assert lib.fake_pinned_blocks() == kept
    assert lib.fake_device_blocks() == before


def generation(lib, rows, cols, **kw):
    """The launches of the second of two generations of a bitmap search."""
    base = dict(pop_size=100, max_len=20, init_max_len=20, elite=2, n_biclusters=3, mode=2,
                tabu_hit_limit=0, neg_trends=1, ratio_num=85, ratio_den=100, use_graph=0)
    base.update(kw)
    p = lib.ebic.Params.make(**base)
    ctx = lib.context()
    assert lib.load(ctx, rows, cols) == 0 and lib.run(ctx, p, 1)[0] == 0
    lib.fake_clear_log()
    assert lib.run(ctx, p, 1)[0] == 0
    lib.ebic_destroy(ctx)
    return [k for k, _ in lib.log()]


@pytest.mark.parametrize("rows,pop,attempts,ratio,max_len,block", [
    (10_000, 800, 4, (85, 100), 20, 1), (13_579, 800, 4, (85, 100), 20, 1),   # the usual searches
    (8192, 100, 4, (1, 2), 64, 1), (8193, 100, 4, (1, 2), 12, 0),              # long children
    (8192, 1200, 4, (3, 4), 20, 1), (16_000, 1200, 4, (4, 5), 20, 0),
    (32_768, 100, 4, (85, 100), 20, 1), (32_768, 100, 4, (85, 100), 64, 0),    # few warps
    (33_000, 100, 4, (85, 100), 20, 0), (50_000, 456, 4, (9, 10), 20, 0),
    (60_000, 800, 4, (85, 100), 20, 1), (60_000, 800, 4, (85, 100), 64, 0),    # many warps
    (40_000, 800, 4, (85, 100), 64, 1), (65_536, 1200, 4, (85, 100), 41, 1),
    (65_537, 1200, 4, (85, 100), 20, 0), (16_384, 1200, 4, (1, 1), 64, 1),
    (49_152, 100, 4, (1, 1), 20, 1), (50_000, 100, 4, (1, 1), 20, 0),
    (16_384, 100, 1, (85, 100), 20, 0), (8192, 100, 1, (85, 100), 20, 1)])
def test_small_searches_evaluate_in_the_evolve_launch_where_it_pays(lib, rows, pop, attempts, ratio,
                                                                     max_len, block):
    ran = generation(lib, rows, 30 if max_len < 30 else 64, pop_size=pop, max_attempts=attempts,
                     ratio_num=ratio[0], ratio_den=ratio[1], max_len=max_len, init_max_len=max_len)
    assert any("k_evolve_block" in k for k in ran) == bool(block)
    assert sum("k_eval" in k for k in ran) == 1 - block


@pytest.mark.parametrize("rows,pop,ratio,fuse,one", [
    (4500, 96, (85, 100), -1, 0), (4500, 96, (1, 2), -1, 1), (4500, 96, (85, 100), 2, 1),
    (4500, 1400, (9, 10), -1, 0), (60_000, 1200, (85, 100), -1, 0), (60_000, 1300, (85, 100), -1, 1),
    (20_000, 4096, (85, 100), -1, 1), (16_000, 4096, (1, 1), -1, 0)])
def test_generations_read_one_direction_where_it_pays(lib, rows, pop, ratio, fuse, one):
    """No tied pairs: a generation's evaluation over every slot takes the one-direction form from
    19,456 passes on, over a list or at a low ratio always (an exact ratio has no staged form)."""
    def count(kernel, grid, args):
        if "k_count_tied" in kernel:
            ints(words(args[3], 1)[0], 1)[0] = 0

    lib.hook(count)
    ran = generation(lib, rows, 700, pop_size=pop, ratio_num=ratio[0], ratio_den=ratio[1],
                     fuse_pairs=fuse)
    used = [k for k in ran if "k_eval_bitmap" in k]
    assert len(used) == 1
    assert ("k_eval_bitmap_one" in used[0]) == bool(one)


@pytest.mark.parametrize("rows,entries,waits", [(10_000, 20, 1), (10_000, 100, 1), (10_000, 256, 2),
                                                (33_333, 100, 2)])
def test_large_masks_are_not_copied_twice(lib, rows, entries, waits):
    """Masks of up to 160 KB for the whole list come with the counters in one wait; larger ones, of the
    entries there are, straight to the caller after the count."""
    p = lib.ebic.Params.make(pop_size=300, max_len=6, init_max_len=6, elite=2, n_biclusters=entries,
                             mode=1)
    ctx = lib.context()
    assert lib.load(ctx, rows, 20) == 0 and lib.run(ctx, p, 1)[0] == 0
    out = np.zeros((256, (rows + 127) // 128 * 4), np.uint32)
    n = ctypes.c_int32()
    for _ in range(2):                                # (the first call makes the buffer)
        lib.fake_clear_log()
        assert lib.ebic_extract_biclusters(ctx, 256, out.ctypes.data, ctypes.byref(n)) == 0
    assert lib.fake_calls(b"synchronise") == waits
    lib.ebic_destroy(ctx)
