"""GPU tests of the hit kernel's passes and of the table build: tickets of
every size over tasks of one hit (many passes of 32 tasks to a ticket) and of
thousands (a pass of one task), and tables rebuilt by an update of the weights
or the fractions alone.  Deterministic mode is bit-exact against the oracle's
canonical fold, so every cell checks every hit's bin and cell."""
import dataclasses

import numpy as np
import pytest

from oracle import oracle as O
from paper_2103_14737_gb300 import fcs, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("hit_E", [(2.0e4, 1.0e5), (0.05, 0.2)])  # about one hit a task; up to thousands
def test_tickets(geo, ogeo, hit_E):
    prm = synth.params(geo, mean_hit_range=hit_E)
    parts = synth.ttbar_like(4, 2, n=150 if hit_E[0] > 1.0 else 8)
    ref = O.simulate(ogeo, O.OracleParams(prm), parts, seed=9)
    s = fcs.Simulator(geo, prm)
    try:
        d = s.to_device(parts)
        for hpt in (0, 1, 2, 4, 8):
            for block in (0, 256, 512):
                got = s.simulate(d, 9, mode=fcs.MODE_DETERMINISTIC, dense=True, hits_per_thread=hpt, block=block)
                assert got["stats"]["n_hits"] == ref.n_hits
                assert np.array_equal(got["cells"].cpu().numpy().view(np.uint32), ref.cells_canon.view(np.uint32)), (hpt, block)
                atom = s.simulate(d, 9, dense=True, hits_per_thread=hpt, block=block)["cells"].cpu().numpy()
                assert (np.abs(atom - ref.cells64) <= 1e-5 * np.abs(ref.cells64) + 1e-3).all()
    finally:
        s.close()


def test_table_updates(geo, prm, ogeo):
    """Weights updated while some fractions are 0, then the fractions alone:
    the entries that come alive have tables of the present weights."""
    parts = synth.ttbar_like(3, 1)
    rng = np.random.default_rng(2)
    off = rng.random(prm.frac.shape) < 0.5
    off[..., 0] = False
    off[..., 4] = False
    frac0 = np.where(off, 0.0, prm.frac).astype(np.float32)
    w1 = (prm.shape_w * (0.5 + rng.random(prm.shape_w.shape))).astype(np.float32)
    s = fcs.Simulator(geo, dataclasses.replace(prm, frac=frac0))
    try:
        d = s.to_device(parts)

        def check(p):
            ref = O.simulate(ogeo, O.OracleParams(p), parts, 5)
            det = s.simulate(d, 5, mode=fcs.MODE_DETERMINISTIC, dense=True)["cells"].cpu().numpy()
            assert np.array_equal(det.view(np.uint32), ref.cells_canon.view(np.uint32))

        def dev(a):
            return torch.as_tensor(np.ascontiguousarray(a), device="cuda").reshape(-1)

        check(dataclasses.replace(prm, frac=frac0))
        s.update_params(frac=dev(prm.frac))  # entries that were off at the load
        check(prm)
        s.update_params(frac=dev(frac0), shape_w=dev(w1))
        check(dataclasses.replace(prm, frac=frac0, shape_w=w1))
        s.update_params(frac=dev(prm.frac))  # entries that were off when the weights came
        check(dataclasses.replace(prm, shape_w=w1))
    finally:
        s.close()


def test_backward_outgrows_workspace(geo, prm):
    """A synchronous backward call on a workspace sized by a smaller call runs
    again with the workspace grown: the gradients are those of a fresh one."""
    small, big = synth.single_particle(1), synth.ttbar_like(3, 4)
    out = []
    for first in (small, big):
        s = fcs.Simulator(geo, prm)
        try:
            g = torch.Generator("cuda").manual_seed(1)
            dl = torch.randn((4, s.n_cells), generator=g, device="cuda")
            s.backward(s.to_device(first), 3, dl[:first.n_events])
            r = s.backward(s.to_device(big), 3, dl)
            torch.cuda.synchronize()
            assert r["status"] == 0
            out.append((r["stats"], r["d_frac"].cpu(), r["d_shape_w"].cpu()))
        finally:
            s.close()
    assert out[0][0]["n_hits"] == out[1][0]["n_hits"] > 0
    for a, b in zip(out[0][1:], out[1][1:]):
        torch.testing.assert_close(a, b, rtol=1e-6, atol=1e-6 * float(b.abs().max()))


@pytest.mark.parametrize("n_events, share", [(32, 1), (33, 8), (310, 2), (64, 0), (305, -1)])
def test_sparse_events(geo, prm, ogeo, n_events, share):
    """Calls of at least 32 events and at most 8 particles an event read back
    only the cells that their deposits marked: the same pairs as a call that
    reads every cell, over empty events, an event with every particle (-1),
    event ranges, graphs and outputs that are too small, and rows left zero."""
    rng = np.random.default_rng(n_events)
    n = max(share, 1) * n_events
    off = np.arange(n_events + 1, dtype=np.int64) * share if share > 0 else np.where(
        np.arange(n_events + 1) > (n_events // 2 if share < 0 else 0), n, 0).astype(np.int64)
    if share == 0:  # every second event empty
        off = np.minimum((np.arange(n_events + 1) + 1) // 2 * 2, n).astype(np.int64)
    parts = synth.Particles(rng.integers(0, 3, n).astype(np.int32), rng.uniform(1e3, 1e5, n).astype(np.float32),
                            rng.uniform(-5.2, 5.2, n).astype(np.float32), rng.uniform(-3.2, 3.2, n).astype(np.float32),
                            off)
    oracle = O.simulate(ogeo, O.OracleParams(prm), parts, seed=4)
    ref, canon = oracle.cells64, oracle.cells_canon
    s = fcs.Simulator(geo, prm)
    try:
        d = s.to_device(parts)

        def check(r, n_read=None):
            eo = r["event_offsets"].cpu().numpy()
            nnz = int(eo[-1]) if n_read is None else n_read
            ids, E = r["cell_ids"][:nnz].cpu().numpy(), r["cell_E"][:nnz].cpu().numpy()
            ev, cell = np.nonzero(ref)
            assert np.array_equal(eo, np.searchsorted(ev, np.arange(n_events + 1)))
            assert np.array_equal(ids, cell[:nnz])
            np.testing.assert_allclose(E, ref[ev, cell][:nnz], rtol=1e-5)

        general = s.simulate(d, 4, debug_hits=1, capacity=1 << 18)  # reads every cell
        check(general)
        check(s.simulate(d, 4))
        check(s.simulate(d, 4, block=256))
        check(s.simulate(d, 4, block=512, wave_events=40))
        nnz = int(general["event_offsets"][-1])
        small = s.simulate(d, 4, capacity=nnz - 3, check=False)
        assert small["status"] == fcs.FCS_E_RANGE
        check(small, nnz - 3)
        out = {k: general[k] for k in ("cell_ids", "cell_E", "event_offsets")}
        for _ in range(2):  # captured, replayed
            out["cell_ids"].fill_(-1)
            s.simulate(d, 4, sync=0, use_graph=1, outputs=out)
            torch.cuda.synchronize()
            check(out)
        pin = [torch.as_tensor(a).pin_memory() for a in (parts.type, parts.E, parts.eta, parts.phi, parts.event_offsets)]
        host = {k: torch.zeros(v.shape, dtype=v.dtype).pin_memory() for k, v in out.items()}
        for _ in range(2):  # host buffers, in waves of events
            host["cell_ids"].fill_(-1)
            fcs.fcs_simulate_events_host(s.geo, s.prm, s.ws, *(a.numpy() for a in pin), 4, 0, fcs.make_config(),
                                         *(host[k].numpy() for k in ("cell_ids", "cell_E", "event_offsets")))
            check(host)
        det = fcs.MODE_DETERMINISTIC  # the canonical fold, bit for bit
        for r in (s.simulate(d, 4, mode=det), s.simulate(d, 4, mode=det, wave_events=40),
                  s.simulate(d, 4, mode=det, debug_hits=1), s.simulate(d, 4, mode=det, block=256)):
            check(r)
            ev, cell = np.nonzero(ref)
            assert np.array_equal(r["cell_E"][:nnz].cpu().numpy().view(np.uint32), canon[ev, cell].view(np.uint32))
        for mode in (fcs.MODE_ATOMIC, det):  # the dense rows too, all of them written
            dense = dict(out, cells=torch.full((n_events, s.n_cells), -1.0, device="cuda"))
            check(s.simulate(d, 4, mode=mode, outputs=dense))
            want = torch.zeros_like(dense["cells"])
            ev, cell = (torch.as_tensor(a, device="cuda") for a in np.nonzero(ref))
            want[ev, cell] = dense["cell_E"][:nnz]
            assert torch.equal(dense["cells"], want)
            only = s.simulate(d, 4, mode=mode, outputs=dict(cells=torch.full_like(want, -1.0)), wave_events=40)["cells"]
            torch.testing.assert_close(only, want, rtol=1e-5, atol=1e-3)
        check(s.simulate(d, 4, debug_hits=1, capacity=1 << 18))  # the rows were left zero
    finally:
        s.close()


@pytest.mark.parametrize("n, E", [(1, 1.0e6), (3, 3.0e5), (340, 3.0e3), (380, 3.0e3), (1500, 1.0e4)])
def test_long_segments(geo, prm, ogeo, n, E):
    """Cells of many records in deterministic mode: few tasks with thousands of
    records, about as many tasks as the fold's table takes, and more than that
    with fewer and with more than 1024 records."""
    parts = synth.Particles(np.zeros(n, np.int32), np.full(n, E, np.float32), np.full(n, 0.22, np.float32),
                            np.zeros(n, np.float32), np.array([0, n], np.int64))
    canon = O.simulate(ogeo, O.OracleParams(prm), parts, seed=6).cells_canon
    s = fcs.Simulator(geo, prm)
    try:
        got = s.simulate(s.to_device(parts), 6, mode=fcs.MODE_DETERMINISTIC, dense=True)["cells"].cpu().numpy()
        assert np.array_equal(got.view(np.uint32), canon.view(np.uint32))
    finally:
        s.close()


@pytest.mark.parametrize("n, E_first", [(90_000, 500.0), (90_001, 1.5e8), (91_351, 500.0)])
def test_long_task_lists(geo, prm, ogeo, n, E_first):
    """The hit offsets of more than 2^21 possible tasks: remainders of the lanes'
    four tasks and of the warps', and a task of more than 2^21 hits, whose warp
    adds in 64 bits."""
    rng = np.random.default_rng(n)
    E = rng.uniform(50.0, 500.0, n).astype(np.float32)
    E[n // 3] = E_first
    parts = synth.Particles(rng.integers(0, 3, n).astype(np.int32), E, rng.uniform(-4.0, 4.0, n).astype(np.float32),
                            rng.uniform(-3.1, 3.1, n).astype(np.float32), np.array([0, n // 2, n], np.int64))
    parts.eta[n // 3], parts.type[n // 3] = 0.2, 0
    ref = O.simulate(ogeo, O.OracleParams(prm), parts, seed=3)
    s = fcs.Simulator(geo, prm)
    try:
        got = s.simulate(s.to_device(parts), 3, mode=fcs.MODE_DETERMINISTIC, dense=True)
        assert got["stats"]["n_hits"] == ref.n_hits and got["stats"]["n_tasks"] == ref.n_tasks
        assert np.array_equal(got["cells"].cpu().numpy().view(np.uint32), ref.cells_canon.view(np.uint32))
    finally:
        s.close()


def test_host_calls_with_new_arguments(geo, prm):
    """Host-buffer calls on one workspace whose seeds, first events, event counts,
    number of waves and density change from call to call, each against a device
    call: the instantiated graph takes the new parameters or is made anew."""
    batches = [synth.pileup(3, 5, mu_pu=20), synth.pileup(4, 6, mu_pu=20), synth.pileup(5, 2, mu_pu=20),
               synth.single_particle(70), synth.single_particle(520)]
    s, h = fcs.Simulator(geo, prm), fcs.Simulator(geo, prm)
    try:
        cap = 1 << 19
        out = [torch.zeros(cap, dtype=torch.int32).pin_memory(), torch.zeros(cap).pin_memory()]
        for k, (i, seed, first) in enumerate([(1, 9, 0), (0, 1, 0), (0, 2, 0), (0, 2, 7), (1, 2, 7), (2, 3, 0), (0, 1, 0),
                                              (3, 1, 0), (3, 2, 0), (4, 1, 0), (4, 5, 1), (0, 1, 0)]):
            parts = batches[i]
            pin = [torch.as_tensor(a).pin_memory().numpy()
                   for a in (parts.type, parts.E, parts.eta, parts.phi, parts.event_offsets)]
            off = torch.zeros(parts.n_events + 1, dtype=torch.int64).pin_memory()
            out[0].fill_(-1)
            fcs.fcs_simulate_events_host(h.geo, h.prm, h.ws, *pin, seed, first, fcs.make_config(), out[0].numpy(),
                                         out[1].numpy(), off.numpy())
            ref = s.simulate(s.to_device(parts), seed, first_event=first, capacity=cap)
            nnz = int(off[-1])
            assert torch.equal(off, ref["event_offsets"].cpu()), k
            assert torch.equal(out[0][:nnz], ref["cell_ids"][:nnz].cpu()), k
            torch.testing.assert_close(out[1][:nnz], ref["cell_E"][:nnz].cpu(), rtol=1e-5, atol=1e-3)
    finally:
        s.close()
        h.close()
