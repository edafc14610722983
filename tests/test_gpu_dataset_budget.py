"""Datasets under a device-memory budget (rs_set_dataset_budget): least recently used datasets not
in use are evicted and rebuilt from the host copy when next named; every count stays equal to the
oracle's, through cached graphs, asynchronous calls and serving requests that pin their dataset."""
import ctypes

import numpy as np
import pytest

from paper_2406_01821_gb300 import synth

pytestmark = pytest.mark.gpu

N, F, K = 4000, 12, 3


def _data(i):
    X, y = synth.gaussian_mixture(N, F, K, 60 + i)
    b = synth.random_rulesets(synth.quantile_table(X), K, 40, (1, 12), (1, 4), 70 + i, pair_prob=0.3)
    return X, y, b


def _budget_ctx(flags=0):
    """A context whose budget holds two of the test's (equally sized) datasets."""
    from paper_2406_01821_gb300 import build, rs
    build.build()
    ctx = rs.Context(0, flags=flags)
    ctx.set_dataset_budget(1 << 40)             # keep host copies from the first registration on
    return ctx


def test_evict_least_recently_used_and_rebuild(orc):
    from paper_2406_01821_gb300 import rs
    ctx = _budget_ctx()
    try:
        data = [_data(i) for i in range(3)]
        want = [orc.eval_hard(X, y, K, b) for X, y, b in data]
        dss = [ctx.dataset(data[0][0], data[0][1], K)]
        one = ctx.dataset_stats()["resident_bytes"]
        ctx.set_dataset_budget(2 * one + one // 2)
        dss += [ctx.dataset(X, y, K) for X, y, _ in data[1:]]
        st = ctx.dataset_stats()
        assert st["datasets"] == 3 and st["resident"] == 2 and st["evictions"] == 1     # the first
        assert st["resident_bytes"] <= 2 * one + one // 2

        def check(i):
            c, pc, _ = ctx.eval_hard(dss[i], rs.HostBatch(data[i][2]), K)
            assert np.array_equal(c, want[i][0]) and np.array_equal(pc, want[i][1].reshape(-1, K))

        check(0)                                   # rebuilt; the second is now least recent
        st = ctx.dataset_stats()
        assert st["rebuilds"] == 1 and st["evictions"] == 2 and st["resident"] == 2
        check(2)                                   # resident: nothing moves
        assert ctx.dataset_stats()["rebuilds"] == 1
        check(1)                                   # rebuilt, the first evicted again
        st = ctx.dataset_stats()
        assert st["rebuilds"] == 2 and st["evictions"] == 3
        # device batches repeat on one stream (cached and captured graphs), around an eviction
        import torch
        stream = torch.cuda.Stream()
        db = rs.DeviceBatch.from_host(data[0][2])
        for rnd in range(2):
            for _ in range(3):
                c, pc, _ = ctx.eval_hard(dss[0], db, K, stream=stream)
                stream.synchronize()
                assert np.array_equal(c.cpu().numpy(), want[0][0])
            check(1)
            check(2)                               # the first is evicted between the rounds
        assert ctx.dataset_stats()["evictions"] >= 5
        ctx.dataset_destroy(dss[0])                # whether resident or not
        st = ctx.dataset_stats()
        assert st["datasets"] == 2
    finally:
        ctx.close()


def test_async_calls_and_static_entry(orc):
    import torch
    from paper_2406_01821_gb300 import rs
    ctx = _budget_ctx(flags=rs.CTX_ASYNC)
    try:
        data = [_data(i) for i in range(3)]
        want = [orc.eval_hard(X, y, K, b) for X, y, b in data]
        dss = [ctx.dataset(data[0][0], data[0][1], K)]
        one = ctx.dataset_stats()["resident_bytes"]
        ctx.set_dataset_budget(2 * one + one // 2)
        dss.append(ctx.dataset(data[1][0], data[1][1], K))
        stream = torch.cuda.Stream()
        dbs = [rs.DeviceBatch.from_host(b) for _, _, b in data]
        outs = []
        for i in (0, 1):                           # enqueued, not waited for
            c = torch.empty(dbs[i].c().P, dtype=torch.int32, device="cuda")
            pc = torch.empty((dbs[i].c().P, K), dtype=torch.int32, device="cuda")
            ctx.eval_hard(dss[i], dbs[i], K, out=(c, pc, None), stream=stream)
            outs.append((c, pc))
        # a dataset whose queued work has not completed is not evicted (its mark is pending);
        # whichever is chosen, the queued results are exact
        dss.append(ctx.dataset(data[2][0], data[2][1], K))
        rs.check(rs.lib().rs_check(ctx.h, rs._stream_ptr(stream)))
        for i in (0, 1):
            assert np.array_equal(outs[i][0].cpu().numpy(), want[i][0])
            assert np.array_equal(outs[i][1].cpu().numpy(), want[i][1].reshape(-1, K))
        assert ctx.dataset_stats()["evictions"] <= 1
        if ctx.dataset_stats()["resident"] == 3:     # nothing was idle then: make room now
            c, _, _ = ctx.eval_hard(dss[2], rs.HostBatch(data[2][2]), K)
            ctx.set_dataset_budget(2 * one + one // 2)
        assert ctx.dataset_stats()["resident"] == 2
        for i in (2, 1):                           # synchronous uses: the first is left evicted
            c = torch.empty(dbs[i].c().P, dtype=torch.int32, device="cuda")
            ctx.eval_hard(dss[i], dbs[i], K, out=(c, None, None), stream=stream)
            rs.check(rs.lib().rs_check(ctx.h, rs._stream_ptr(stream)))
            assert np.array_equal(c.cpu().numpy(), want[i][0])
        assert ctx.dataset_stats()["resident"] == 2
        # the allocation-free entry refuses an evicted dataset (rebuilding would allocate)
        cb = dbs[0].c()
        c = torch.empty(cb.P, dtype=torch.int32, device="cuda")
        pc = torch.empty((cb.P, K), dtype=torch.int32, device="cuda")
        rc = rs.lib().rs_eval_hard_static(ctx.h, dss[0], ctypes.byref(cb), rs._ptr(c), rs._ptr(pc), None,
                                          rs._stream_ptr(stream))
        assert rc == -1                            # RS_ERR_INVALID
        ctx.eval_hard(dss[0], dbs[0], K, out=(c, pc, None), stream=stream)   # rebuilt
        rc = rs.lib().rs_eval_hard_static(ctx.h, dss[0], ctypes.byref(cb), rs._ptr(c), rs._ptr(pc), None,
                                          rs._stream_ptr(stream))
        assert rc == 0
        rs.check(rs.lib().rs_check(ctx.h, rs._stream_ptr(stream)))
        assert np.array_equal(c.cpu().numpy(), want[0][0])
    finally:
        ctx.close()


def test_serving_request_pins_its_dataset(orc):
    from paper_2406_01821_gb300 import rs
    ctx = _budget_ctx()
    try:
        data = [_data(i) for i in range(4)]
        want = [orc.eval_hard(X, y, K, b) for X, y, b in data]
        dss = [ctx.dataset(data[0][0], data[0][1], K)]
        one = ctx.dataset_stats()["resident_bytes"]
        ctx.set_dataset_budget(2 * one + one // 2)
        dss.append(ctx.dataset(data[1][0], data[1][1], K))
        ticket = ctx.submit(dss[0], rs.HostBatch(data[0][2]))   # pins the first until polled
        dss += [ctx.dataset(X, y, K) for X, y, _ in data[2:]]   # would evict the first otherwise
        for i in (2, 3, 1, 2, 3):
            c, _, _ = ctx.eval_hard(dss[i], rs.HostBatch(data[i][2]), K)
            assert np.array_equal(c, want[i][0])
        rebuilds = ctx.dataset_stats()["rebuilds"]
        c, pc, _ = ctx.poll(ticket, data[0][2].P, K, timeout_us=60_000_000)
        assert np.array_equal(c, want[0][0]) and np.array_equal(pc, want[0][1].reshape(-1, K))
        c, _, _ = ctx.eval_hard(dss[0], rs.HostBatch(data[0][2]), K)
        assert np.array_equal(c, want[0][0])
        assert ctx.dataset_stats()["rebuilds"] == rebuilds      # it was never evicted
    finally:
        ctx.close()


def test_work_queued_without_a_budget_is_waited_for(orc):
    """A dataset with a host copy, used by an asynchronous call while no budget is set: a budget set
    before that work has run does not take the memory from under it."""
    import torch
    from paper_2406_01821_gb300 import rs
    ctx = _budget_ctx(flags=rs.CTX_ASYNC)
    try:
        (X, y, b), (X2, y2, _) = _data(0), _data(1)
        want = orc.eval_hard(X, y, K, b)
        ds = ctx.dataset(X, y, K)
        ctx.set_dataset_budget(0)
        db = rs.DeviceBatch.from_host(b)
        stream = torch.cuda.Stream()
        c = torch.empty(b.P, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            torch.cuda._sleep(200_000_000)         # some 0.1 s before the call's kernels
        ctx.eval_hard(ds, db, K, out=(c, None, None), stream=stream)
        ctx.set_dataset_budget(1)
        assert not stream.query() and ctx.dataset_stats()["evictions"] == 0
        other = ctx.dataset(X2, y2, K)             # would take the evicted dataset's place
        rs.check(rs.lib().rs_check(ctx.h, rs._stream_ptr(stream)))
        assert np.array_equal(c.cpu().numpy(), want[0])
        ctx.dataset_destroy(other)
        ctx.set_dataset_budget(1)                  # the work has completed: evicted now
        assert ctx.dataset_stats()["evictions"] == 1
    finally:
        ctx.close()


@pytest.mark.parametrize("finite", (True, False))
def test_eviction_under_a_live_serving_kernel(orc, finite):
    """Two datasets of one shape and different labels take each other's place in device memory while
    requests on a third keep the serving kernel running: every request is counted with its own
    dataset's labels and features."""
    from paper_2406_01821_gb300 import rs
    ctx = _budget_ctx()
    try:
        Xc, yc = synth.gaussian_mixture(200_000, 32, 4, 80)
        bc = synth.random_rulesets(synth.quantile_table(Xc[:4000]), 4, 2000, (32, 64), (4, 8), 81)
        third = ctx.dataset(Xc, yc, 4)
        base = ctx.dataset_stats()["resident_bytes"]
        pair = []
        for i, share in enumerate(((0.2, 0.3, 0.5), (0.6, 0.3, 0.1))):
            X, _, b = _data(i)
            y = np.random.default_rng(82 + i).choice(K, N, p=share).astype(np.int32)
            if not finite:
                X[::37, 3] = np.nan
            pair.append((X, y, b, orc.eval_hard(X, y, K, b)))
        dss = [ctx.dataset(pair[0][0], pair[0][1], K)]
        one = ctx.dataset_stats()["resident_bytes"] - base
        ctx.set_dataset_budget(base + one + one // 2)
        dss.append(ctx.dataset(pair[1][0], pair[1][1], K))
        assert ctx.dataset_stats()["resident"] == 2
        dbc = rs.DeviceBatch.from_host(bc)
        backlog = [ctx.submit(third, dbc) for _ in range(24)]
        for rnd in range(12):
            i = rnd & 1
            _, _, b, want = pair[i]
            out = ctx.poll(ctx.submit(dss[i], rs.HostBatch(b)), b.P, K, timeout_us=60_000_000)
            assert np.array_equal(out[0], want[0]), rnd
            assert np.array_equal(out[1], want[1].reshape(-1, K)), rnd
        assert ctx.dataset_stats()["rebuilds"] >= 11
        assert ctx.poll(backlog[-1], bc.P, 4, timeout_us=0) is None     # the kernel was busy throughout
        counts = [ctx.poll(t, bc.P, 4, timeout_us=60_000_000)[0] for t in backlog]
        c, _, _ = ctx.eval_hard(third, rs.HostBatch(bc), 4)
        for got in counts:
            assert np.array_equal(got, c)
    finally:
        ctx.close()


def test_a_small_budget_holds_on_to_no_more(orc):
    """Freed dataset memory that a context holds on to counts towards a budget below 256 MiB. 64 MiB
    allow for the pool's granularity and other processes' noise; the dataset takes 0.25 GiB."""
    import torch
    from paper_2406_01821_gb300 import rs
    ctx = _budget_ctx()
    try:
        X, y, b = _data(0)
        want = orc.eval_hard(X, y, K, b)
        small = ctx.dataset(X, y, K)
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        big = ctx.dataset(np.zeros((1 << 19, 96), np.float32), np.zeros(1 << 19, np.int32), 2)
        assert before - torch.cuda.mem_get_info()[0] >= 4 * 96 << 19
        ctx.eval_hard(small, rs.HostBatch(b), K)   # the more recent of the two
        ctx.set_dataset_budget(16 << 20)           # evicts the large one
        assert ctx.dataset_stats()["resident"] == 1
        assert before - torch.cuda.mem_get_info()[0] <= 64 << 20
        c, _, _ = ctx.eval_hard(small, rs.HostBatch(b), K)
        assert np.array_equal(c, want[0])
        ctx.dataset_destroy(big)
    finally:
        ctx.close()


@pytest.mark.parametrize("reject", (False, True))
def test_dropped_dataset_memory_is_given_back(reject):
    """A context keeps at most 256 MiB of dropped datasets' memory mapped (rs.h); the rest is free for
    any other allocator once the dropping (or rejecting) call has returned. 64 MiB allow for what the
    calls load for the first time and other processes' noise; the dataset and its scratch take 0.65 GiB."""
    import torch
    from paper_2406_01821_gb300 import build, rs
    build.build()
    ctx = rs.Context(0)
    try:
        n, f = 1 << 20, 128
        X = torch.zeros((n, f), device="cuda")
        y = torch.zeros(n, dtype=torch.int32, device="cuda")
        if reject:
            y[n // 2] = 7                          # not a class of K = 2
        small = ctx.dataset(np.zeros((300, 4), np.float32), np.zeros(300, np.int32), 2)
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        if reject:
            with pytest.raises(rs.RsError):
                ctx.dataset(X, y, 2)
        else:
            ds = ctx.dataset(X, y, 2)
            assert before - torch.cuda.mem_get_info()[0] >= 4 * n * f
            ctx.dataset_destroy(ds)
        assert before - torch.cuda.mem_get_info()[0] <= (256 + 64) << 20
        ctx.dataset_destroy(small)
    finally:
        ctx.close()
