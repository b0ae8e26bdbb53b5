"""Calls short of device memory: one that fails leaves nothing running and its
context usable, and one that fits by the general path takes it."""
import numpy as np
import pytest

import graphgen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def take_device(hold):
    size = 1 << 37
    while size >= 8 << 20:  # the workspace grows by 64 MB or more
        try:
            hold.append(torch.empty(size, dtype=torch.uint8, device="cuda"))
        except torch.OutOfMemoryError:
            size //= 2


def test_call_without_room_for_its_outputs_returns_after_its_work():
    # Outputs in pageable host memory are staged on the device.  With the whole
    # device taken, the context's workspace (sized by earlier calls with device
    # outputs) has no room for them: the call fails, and by then the stream is
    # idle, so the next call may use the workspace on another stream at once.
    from paper_1205_6693_gb300 import truss as T
    n, rows = 1 << 18, 1 << 22
    s, d = graphgen.rmat_raw_cuda(18, rows, seed=21)
    sup, tr = torch.empty_like(s), torch.empty_like(s)
    ref_sup, ref_tr = torch.empty_like(s), torch.empty_like(s)
    h_sup, h_tr = np.empty(rows, np.int32), np.empty(rows, np.int32)
    # lists from a second walk: the working set does not depend on what is free
    warm = T.Context(0, lists_by_walk=1)  # loads every kernel of the call
    warm.decompose(n, s, d, h_sup, h_tr)
    warm.close()
    ctx = T.Context(0, lists_by_walk=1)
    hold = []
    try:
        for _ in range(2):
            ctx.decompose(n, s, d, ref_sup, ref_tr)
        other = torch.cuda.Stream()
        torch.cuda.synchronize()
        take_device(hold)
        with pytest.raises(T.TrussError) as ei:
            ctx.decompose(n, s, d, h_sup, h_tr)
        idle = torch.cuda.current_stream().query()
        assert ei.value.code == T.TRUSS_ENOMEM
        assert idle
        ctx.decompose(n, s, d, sup, tr, stream=other.cuda_stream)
        hold.clear()
        torch.cuda.empty_cache()
        assert torch.equal(sup, ref_sup) and torch.equal(tr, ref_tr)
    finally:
        hold.clear()
        ctx.close()
        torch.cuda.empty_cache()


def test_small_graph_of_many_duplicates_fits_the_general_paths_workspace():
    # The one-launch build holds arrays for every row, the general path for
    # every distinct edge: with the device taken and a workspace sized by the
    # general path (which a wait limit selects) the call still succeeds.
    from paper_1205_6693_gb300 import truss as T
    n, rows = 30_000, 2_600_000
    gen = torch.Generator(device="cuda").manual_seed(4)
    s, d = (torch.randint(0, 3000, (2600,), dtype=torch.int32, generator=gen,
                          device="cuda").repeat(rows // 2600) for _ in range(2))
    ref_sup, ref_tr = torch.empty_like(s), torch.empty_like(s)
    sup, tr = torch.empty_like(s), torch.empty_like(s)
    warm = T.Context(0)  # loads the kernels of the one-launch build
    warm.decompose(n, s, d, sup, tr)
    warm.close()
    ctx = T.Context(0, wait_limit_ns=4_000_000_000)
    hold = []
    try:
        for _ in range(2):
            k = ctx.decompose(n, s, d, ref_sup, ref_tr)
        torch.cuda.synchronize()
        take_device(hold)
        ctx.set_opts()
        assert ctx.decompose(n, s, d, sup, tr) == k
        hold.clear()
        torch.cuda.empty_cache()
        assert torch.equal(sup, ref_sup) and torch.equal(tr, ref_tr)
    finally:
        hold.clear()
        ctx.close()
        torch.cuda.empty_cache()


@pytest.mark.parametrize("graphs", [1, 100])
def test_workspace_per_vertex_of_the_general_path(graphs):
    # what a vertex adds where vertices outnumber rows: fifteen words, before its
    # degree was sorted with its graph's number
    from paper_1205_6693_gb300 import truss as T
    gen = torch.Generator(device="cuda").manual_seed(1)
    peaks = []
    for n in (4_000_000, 8_000_000):  # above the one-launch build's limit
        s, d = (torch.randint(0, n // graphs, (60_000,), dtype=torch.int32, generator=gen,
                              device="cuda") for _ in range(2))
        sup, tr = torch.empty_like(s), torch.empty_like(s)
        ctx = T.Context(0)
        if graphs == 1:
            ctx.decompose(n, s, d, sup, tr)
        else:
            off = np.arange(graphs + 1, dtype=np.int64) * (60_000 // graphs)
            ctx.decompose_batch(np.full(graphs, n // graphs, np.int64), off, s, d, sup, tr)
        peaks.append(ctx.stats()["workspace_peak"])
        ctx.close()
    assert (peaks[1] - peaks[0]) / 4_000_000 <= 60.2
