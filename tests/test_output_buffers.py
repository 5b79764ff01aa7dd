"""Which results of the device-resident call a later call on the same simulator
may overwrite: records by records, start and completion steps by start and
completion steps, and nothing by a call that returns host arrays of a few
requests."""
import types

import numpy as np
import pytest

from conftest import cuda_available

N, n = 5, 40
TWO = (["fcfs", "isjl"], [0, 9])
SEVEN = (["fcfs", "ljf", "isjl", "isjl", "isjl", "sjf", "isjl_beta"], [0, 0, 0, 9, 40, 0, 9])


def span(t):
    return t.data_ptr(), t.data_ptr() + t.numel() * t.element_size()


def test_records_never_lie_over_steps():
    """The output tensors alone, in host memory: no record of any call lies where
    an earlier call's start or completion steps are."""
    import torch
    from paper_2608_02244_gb300 import sim
    S = object.__new__(sim.Simulator)
    S.n_inst, S.n, S.B, S.handle = N, n, 4, None
    S._records = S._per_req = S._block = None
    S.torch = types.SimpleNamespace(empty=lambda k, dtype, device: torch.empty(k, dtype=dtype),
                                    uint8=torch.uint8, int32=torch.int32)
    for runs in (1, 2, 7, 32):
        _, st, co = S.buffers(runs, True)
        assert span(st)[1] <= span(co)[0] or span(co)[1] <= span(st)[0]
        assert st.numel() == co.numel() == runs * N * n and st.dtype == torch.int32
        for later in (1, 2, 3, 7, 9, 32):
            rec, none, _ = S.buffers(later, False)
            assert none is None and rec.numel() == later * N * sim.RECORD_DTYPE.itemsize
            for t in (st, co):
                assert span(t)[1] <= span(rec)[0] or span(rec)[1] <= span(t)[0], (runs, later)


@pytest.mark.gpu
@pytest.mark.skipif(not cuda_available(), reason="needs a CUDA GPU")
def test_steps_outlive_a_records_only_sweep():
    import torch
    from paper_2608_02244_gb300 import sim
    rng = np.random.default_rng(4)
    a = np.sort(rng.integers(0, 60, (N, n)), axis=1).astype(np.int32)
    p = rng.integers(0, 9, (N, n)).astype(np.int32)
    o = rng.integers(1, 70, (N, n)).astype(np.int32)
    dev = [torch.from_numpy(x).cuda() for x in (a, p, o)]
    S = sim.Simulator(N, n, 4)
    try:
        S.sweep_async(*dev, *SEVEN, 300, per_request=True)             # room for seven runs
        rec, st, co = S.sweep_async(*dev, *TWO, 300, per_request=True)
        start, completion = st.clone(), co.clone()
        rec7, _, _ = S.sweep_async(*dev, *SEVEN, 300)
        records = rec7.clone()
        assert torch.equal(st, start) and torch.equal(co, completion)
        assert torch.equal(rec7[:rec.numel()], rec)                    # records share a buffer
        res = S.sweep(a, p, o, *TWO, 300, per_request=True)            # host arrays of a few requests
        assert torch.equal(st, start) and torch.equal(co, completion) and torch.equal(rec7, records)
        np.testing.assert_array_equal(res["start"].ravel(), start.cpu().numpy())
        np.testing.assert_array_equal(res["completion"].ravel(), completion.cpu().numpy())
    finally:
        S.close()


@pytest.mark.gpu
@pytest.mark.skipif(not cuda_available(), reason="needs a CUDA GPU")
@pytest.mark.parametrize("shift", [-1, 0, 1])
def test_host_arrays_on_both_sides_of_the_one_copy_line(shift):
    """Outputs of up to ONE_COPY_MAX int32 come back in one copy, larger ones in
    one per array: the same results."""
    from paper_2608_02244_gb300 import sim
    words = sim.RECORD_DTYPE.itemsize // 4
    m = (sim.ONE_COPY_MAX // 2 - words) // 2 + shift      # 2 runs of words + 2 m int32
    rng = np.random.default_rng(5)
    o = rng.integers(1, 50, (1, m)).astype(np.int32)
    z = np.zeros_like(o)
    S = sim.Simulator(1, m, 64)
    try:
        both = S.sweep(z, z, o, *TWO, sim.KV_INF, per_request=True)
        assert both["launches"] == 4 and both["status"] == 0
        for i in range(2):
            one = S.sweep(z, z, o, [TWO[0][i]], [TWO[1][i]], sim.KV_INF, per_request=True)
            assert one["records"].tobytes() == both["records"][i].tobytes()
            for f in ("start", "completion"):
                assert one[f].shape == (1, 1, m) and (both[f][i] == one[f][0]).all() and (one[f] >= 0).all()
    finally:
        S.close()


@pytest.mark.parametrize("missing", [0, 1, 2])
def test_a_missing_input_is_refused(missing):
    """The optional counts and slack must not take the place of an input that is
    None: it is refused before anything reaches the device."""
    from paper_2608_02244_gb300 import sim
    import torch
    S = object.__new__(sim.Simulator)
    S.n_inst, S.n, S.B, S.handle, S.torch = N, n, 4, None, torch
    S._records = S._per_req = S._block = None
    x = np.ones((N, n), np.int32)
    args = [None if i == missing else x for i in range(3)]
    with pytest.raises(TypeError):
        S.sweep(*args, *TWO, 300, counts=np.full(N, n, np.int32), slack=x)


@pytest.mark.gpu
@pytest.mark.skipif(not cuda_available(), reason="needs a CUDA GPU")
@pytest.mark.parametrize("copies", [1, 4000])                 # a warp and a thread per task
@pytest.mark.parametrize("max_steps", [0, 25])
def test_start_or_completion_steps_alone(copies, max_steps):
    """Either array may be asked for without the other: every entry is written,
    -1 for what did not start or finish, and the same as with both."""
    import torch
    from paper_2608_02244_gb300 import sim
    rng = np.random.default_rng(8)
    m = 21
    o = np.tile(rng.integers(1, 40, (1, m)), (copies, 1)).astype(np.int32)
    a = np.tile(np.sort(rng.integers(0, 50, (1, m)), axis=1), (copies, 1)).astype(np.int32)
    counts = np.where(np.arange(copies) % 2, m, m - 4).astype(np.int32)
    slack = rng.integers(0, 9, (copies, m)).astype(np.int32)
    a, p, o, counts, slack = (torch.from_numpy(x).cuda() for x in (a, np.zeros_like(o), o, counts, slack))
    R = len(SEVEN[0])
    S = sim.Simulator(copies, m, 3, max_steps=max_steps)
    try:
        for sl in (None, slack):
            got = []
            for want in ((True, True), (True, False), (False, True)):
                rec = torch.empty(R * copies * sim.RECORD_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
                st, co = (torch.full((R, copies, m), -7, dtype=torch.int32, device="cuda") if w else None for w in want)
                rc = sim.isjl_sim_run_sweep(S.handle, *SEVEN, 100, a, p, o, rec, st, co, count=counts, slack=sl)
                assert rc == sim.ISJL_OK
                torch.cuda.synchronize()
                got.append((rec, st, co))
            (rec, st, co), (rec_s, st_s, _), (rec_c, _, co_c) = got
            assert torch.equal(rec, rec_s) and torch.equal(rec, rec_c)
            assert torch.equal(st, st_s) and torch.equal(co, co_c)
            assert int(st.min()) == int(co.min()) == -1                    # the unused slots at least
            if max_steps:
                assert bool(((st >= 0) & (co == -1)).any()) and int(co.max()) <= max_steps
    finally:
        S.close()
