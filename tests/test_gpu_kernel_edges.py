"""The sizes and states at which the step, sampler and training kernels change path: tiles of 128 samples and blocks of
1024 (network, check, training), photons on either side of the plane-wave kernels' pair-rate bound, instance counts
around the step-end kernel's choice of block, tables too large for the rate queues."""
import math

import numpy as np
import pytest
import torch

from oracle import mlp as OM
from paper_2511_08929_gb300 import binding as B
from paper_2511_08929_gb300 import buffers as Q
from paper_2511_08929_gb300 import inputs as I
from paper_2511_08929_gb300 import mlp as GM

pytestmark = pytest.mark.gpu

ETA0 = I.eta0_for_wavelength(0.8)


@pytest.fixture(scope="module")
def tables():
    from paper_2511_08929_gb300 import build as bld
    bld.build()
    t = Q.Tables(chi_min=1e-3, chi_max=1e2, n_chi=24, n_r=64)
    yield t
    t.close()


# ---- photons: the plane-wave kernels against the kernels that read the flags ---------------------------
def _photons(n, seed):
    """Photons from far below any pair rate to far above it, inside and outside the pulse, along and against the
    wave, a few without momentum and a few that are not finite."""
    rng = np.random.default_rng(seed)
    d = rng.normal(size=(n, 3))
    d[: n // 2] = [0.0, 0.0, -1.0] + 0.05 * d[: n // 2]
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    k = np.exp(rng.uniform(math.log(1e-18), math.log(1e6), n))
    k[n // 3:] = np.exp(rng.uniform(math.log(3.0), math.log(3e3), n - n // 3))  # around the bound
    P = np.cross(d, rng.normal(size=(n, 3)))
    P /= np.linalg.norm(P, axis=1, keepdims=True)
    mom = d * k[:, None]
    mom[::97] = 0.0
    pos = np.zeros((n, 3))
    pos[:, 2] = rng.uniform(-20.0, 60.0, n)
    if n > 500:
        pos[251, 2], P[252, 1], mom[253, 0] = np.inf, np.nan, np.nan
    return {"pos": pos, "mom": mom, "spin": P, "w": np.ones(n), "id": np.arange(n, dtype=np.uint64) + 1}


def _pair_steps(tables, b, kind, flags, steps=3):
    n = len(b["id"])
    g = Q.ParticleBuffer(n, B.QED_FP32, B.QED_PHOTON, photons=True)
    g.load(b["pos"], b["mom"], b["spin"], b["w"], b["id"])
    g.init_tau(3)
    e, p = (Q.ParticleBuffer(4 * n + 64, B.QED_FP32, q) for q in (B.QED_ELECTRON, B.QED_POSITRON))
    ctr = Q.Counters()
    f = Q.field(kind, a0=150.0, n_cycles=6.0, phase=2.0, eta0=ETA0)
    for s in range(steps):
        st = Q.step_desc(0.2, 8.0 + 0.2 * s, s, 3, flags=flags)
        B.qed_pair_step(tables.handle, f, st, g.s, e.s, p.s, ctr.ptr)
    c = ctr.read().as_dict()
    c.pop("first_bad")  # the first of several errors is whichever thread came first
    q = g.q.cpu().numpy().view(np.uint32)
    el = e.read()
    order = np.argsort(el["id"])
    return q, {k: v[order] for k, v in el.items()}, c


@pytest.mark.parametrize("kind", [B.QED_FIELD_LP, B.QED_FIELD_CP])
@pytest.mark.parametrize("n", [1, 31, 33, 257, 20011])
def test_pair_rate_bound_changes_nothing(tables, kind, n):
    """T-BMT as printed only concerns leptons, so with that flag beside the full set a photon step is the same
    arithmetic in the kernels that read the flags and have no bound: every word of the photons must agree."""
    b = _photons(n, 40 + n)
    q0, e0, c0 = _pair_steps(tables, b, kind, B.QED_F_FULL)
    q1, e1, c1 = _pair_steps(tables, b, kind, B.QED_F_FULL | B.QED_F_TBMT_PAPER)
    assert c0 == c1
    if n > 1000:
        assert c0["events"] > 0 and c0["nonfinite"] == 9 and 0 < c0["rate_steps"] < 3 * n
    assert np.array_equal(q0, q1)
    for k in e0:
        assert np.array_equal(e0[k], e1[k]), k


def _batch_state(tables, n_inst, flags, steps=4):
    fields = [Q.field((B.QED_FIELD_LP, B.QED_FIELD_CP)[k % 2], a0=150.0 + k % 7, n_cycles=4.0, phase=4 * math.pi, eta0=ETA0)
              for k in range(n_inst)]
    bt = Q.Batch(tables, fields, list(range(5, 5 + n_inst)), [(400, 400, 4000)] * n_inst, 0.2, t0=1.0, flags=flags)
    for k, (e, p, g) in enumerate(bt.buffers()):
        m = (0, 1, 40, 97)[k % 4]
        bm = I.lepton_beam(m, 3000.0, z_range=(-3.0, 3.0), seed=60 + k, id_offset=k << 40)
        e.load(bm["pos"], bm["mom"], bm["spin"], bm["w"], bm["id"])
        bg = _photons(300, 90 + k)
        bg["id"] = bg["id"] + np.uint64((k << 40) + (1 << 30))
        g.load(bg["pos"], bg["mom"], bg["spin"], bg["w"], bg["id"])
        for buf in (e, g):
            if buf.count():
                buf.init_tau(5 + k)
    bt.set_tuning(graph_steps=2)
    bt.step(steps)
    out = []
    for trio in bt.buffers():
        for buf in trio:
            r = buf.read()
            o = np.argsort(r["id"])
            out.append({k: v[o] for k, v in r.items()})
    st, c = bt.stats(), bt.ctr.read().as_dict()
    bt.close()
    c.pop("first_bad")
    return out, (st.step, st.particle_steps, list(st.alive)), c


@pytest.mark.parametrize("n_inst", [1, 32, 33, 300])
def test_step_end_over_instances(tables, n_inst):
    """Counts, compaction and the next plan per instance (8 blocks of 1024 threads up to 32 instances, of 256 above),
    over a graph and a direct remainder, against one batch per instance."""
    out, stats, c = _batch_state(tables, n_inst, None, steps=5)
    assert c["status"] in (0,) and c["events"] > 0 and stats[0] == 5
    again, stats2, c2 = _batch_state(tables, n_inst, None, steps=5)
    assert stats == stats2 and c == c2
    for a, b in zip(out, again):
        for k in a:
            assert np.array_equal(a[k], b[k]), k
    # each instance alone through the single-buffer calls
    for k in sorted({0, 1, 2, n_inst - 1} & set(range(n_inst))):
        f = Q.field((B.QED_FIELD_LP, B.QED_FIELD_CP)[k % 2], a0=150.0 + k % 7, n_cycles=4.0, phase=4 * math.pi, eta0=ETA0)
        e, p = (Q.ParticleBuffer(400, B.QED_FP32, q, use_begin=True) for q in (B.QED_ELECTRON, B.QED_POSITRON))
        g = Q.ParticleBuffer(4000, B.QED_FP32, B.QED_PHOTON, photons=True, use_begin=True)
        m = (0, 1, 40, 97)[k % 4]
        bm = I.lepton_beam(m, 3000.0, z_range=(-3.0, 3.0), seed=60 + k, id_offset=k << 40)
        e.load(bm["pos"], bm["mom"], bm["spin"], bm["w"], bm["id"])
        bg = _photons(300, 90 + k)
        bg["id"] = bg["id"] + np.uint64((k << 40) + (1 << 30))
        g.load(bg["pos"], bg["mom"], bg["spin"], bg["w"], bg["id"])
        for buf in (e, g):
            if buf.count():
                buf.init_tau(5 + k)
        ws, ctr = Q.CompactWorkspace(4000), Q.Counters()
        for s in range(5):
            st = Q.step_desc(0.2, 1.0 + float(s) * 0.2, s, 5 + k)
            B.qed_snapshot_counts([e.s, p.s, g.s])
            B.qed_pair_step(tables.handle, f, st, g.s, e.s, p.s, ctr.ptr)
            B.qed_push_step(tables.handle, f, st, e.s, g.s, ctr.ptr)
            B.qed_push_step(tables.handle, f, st, p.s, g.s, ctr.ptr)
            B.qed_compact(g.s, ws.ptr, ws.bytes)
        for buf, got in zip((e, p, g), out[3 * k:3 * k + 3]):
            r = buf.read()
            o = np.argsort(r["id"])
            for key in r:
                assert np.array_equal(r[key][o], got[key]), (k, key)


def test_tables_beyond_the_rate_queues():
    """A chi grid whose rate tables leave no room for the rate queues runs the kernels that read the flags."""
    t = Q.Tables(chi_min=1e-3, chi_max=1e2, n_chi=9800, n_r=8)
    b = _photons(3001, 7)
    q0, e0, c0 = _pair_steps(t, b, B.QED_FIELD_CP, B.QED_F_FULL)
    q1, e1, c1 = _pair_steps(t, b, B.QED_FIELD_CP, B.QED_F_FULL | B.QED_F_TBMT_PAPER)
    assert c0 == c1 and np.array_equal(q0, q1) and c0["events"] > 0
    out, stats, c = _batch_state(t, 3, None)
    assert stats[0] == 4 and c["events"] > 0
    t.close()


# ---- learned sampler ---------------------------------------------------------------------------------
def _query(n, seed):
    rng = np.random.default_rng(seed)
    to = lambda v: torch.tensor(v, dtype=torch.float64, device="cuda")  # noqa: E731
    r = rng.uniform(0, 1, n)
    r[::11], r[1::13] = 10.0 ** rng.uniform(-14, -2, len(r[::11])), 1.0 - 10.0 ** rng.uniform(-12, -2, len(r[1::13]))
    return to(np.exp(rng.uniform(math.log(2e-3), math.log(5e1), n))), to(r), to(rng.uniform(-1, 1, n))


@pytest.mark.parametrize("n", [1, 127, 129, 1023, 1025, 4097])
def test_sampler_does_not_depend_on_the_launch(tables, n):
    """Every sample is its own: the first n of a larger call, an output array off the 16-byte grid."""
    chi, r, s = _query(200003, 3)
    smp = GM.Sampler(GM.init_params(4))  # untrained: samples that pass, fail and lie in between
    for kw in ({}, {"table_only": True}):
        big, fell, _ = smp.sample(tables, chi, r, s, tol=3e-3, **kw)
        out, f2, nf = smp.sample(tables, chi[:n].contiguous(), r[:n].contiguous(), s[:n].contiguous(), tol=3e-3, **kw)
        assert torch.equal(out, big[:n]) and torch.equal(f2, fell[:n]) and int(nf) == int(f2.sum())
        raw = torch.zeros(4 * n + 1, dtype=torch.float32, device="cuda")
        B.qed_mlp_sample(smp.handle, tables.handle, chi.data_ptr(), r.data_ptr(), s.data_ptr(), n, 3e-3,
                         B.QED_MLP_ALWAYS_TABLE if kw else 0, raw.data_ptr() + 4)
        assert torch.equal(raw[1:].reshape(n, 4), out)
    smp.close()


@pytest.mark.parametrize("n", [1, 127, 129, 20000])
def test_gradient_tiles(tables, n):
    """Partly filled tiles, and more tiles than blocks, against the oracle at the bar of the standard batch (BF16
    roundings next to a boundary: 1e-2 in the norm of a parameter block)."""
    flat = GM.init_params(6)
    smp = GM.Sampler(flat, max_batch=20000)
    x, y, _ = GM.targets(tables, n, 5, 0)
    g, loss = smp.grad(x, y)
    L, gr = OM.loss_and_grads(GM.unflatten(smp.params().astype(np.float64)), x.cpu().numpy().astype(np.float64),
                              y.cpu().numpy().astype(np.float64))
    assert float(loss.item()) == pytest.approx(L, rel=1e-3 if n == 1 else 1e-4)
    gg = GM.unflatten(g.cpu().numpy())
    for k in gr:
        assert np.linalg.norm(gg[k] - gr[k]) <= 1e-2 * max(np.linalg.norm(gr[k]), 1e-30), k
    smp.close()


def test_training_chunks_and_single_steps_agree(tables):
    """Targets generated for several steps at a time are those of the steps: one call of 19 steps of 5000 samples (13
    per chunk) against the loop written out, within the FP32 order of the gradient sums."""
    a, b = (GM.Sampler(GM.init_params(9), max_batch=5000) for _ in range(2))
    loss = a.train(tables, 19, batch=5000, seed=4, lr=1e-3, lr_final=1e-3, weight_decay=0.0)
    for k in range(19):
        x, y, _ = GM.targets(tables, 5000, 4, 5000 * k)
        g, l = b.grad(x, y)
        b.adamw(g, 1e-3, 0.0)
        assert float(l) == pytest.approx(float(loss[k]), rel=1e-4)
    assert np.abs(a.params() - b.params()).max() < 2e-4
    a.close()
    b.close()


@pytest.mark.parametrize("n", [1, 1024, 400003])
def test_sampler_above_the_grid(tables, n):
    """Uniforms within 2e-9 of 1 (a logit above the grid) take the bracketing solver, up to several blocks' queues full
    of them: every one is what it is in a call of its own kind, and between the two branch quantiles' ends."""
    chi, r, s = _query(n, 8)
    top = torch.arange(n, device="cuda") % 3 == 0
    r = torch.where(top, 1.0 - 1.9e-9 * (r * 0.999 + 0.0005), r).contiguous()
    smp = GM.Sampler(GM.init_params(4))
    out, fell, nf = smp.sample(tables, chi, r, s, table_only=True)
    assert bool(torch.isfinite(out).all()) and bool(fell.all()) and int(nf) == n
    alone, _, _ = smp.sample(tables, chi[top].contiguous(), r[top].contiguous(), s[top].contiguous(), table_only=True)
    rest, _, _ = (smp.sample(tables, chi[~top].contiguous(), r[~top].contiguous(), s[~top].contiguous(), table_only=True)
                  if n > 1 else (out[:0], None, None))
    assert torch.equal(out[top], alone) and torch.equal(out[~top], rest)
    smp.close()


def test_sampler_over_many_tiles_a_block(tables):
    """Ten tiles of 1024 samples per block of the check, about a third of whose samples wait in the block's queue, so
    that it fills up between tiles at every offset: each sample is what it is in calls of one tile per block, in which
    the queue never fills."""
    n = 10 * 1024 * torch.cuda.get_device_properties(0).multi_processor_count + 77
    chi, r, s = _query(n, 12)
    smp = GM.Sampler(GM.init_params(4))
    for tol in (3e-3, 2e-2):
        out, fell, nf = smp.sample(tables, chi, r, s, tol=tol)
        assert int(nf) == int(fell.sum()) and 0 < int(nf) < n
        for a in range(0, n, 100000):
            part = slice(a, min(n, a + 100000))
            o1, f1, _ = smp.sample(tables, chi[part], r[part], s[part], tol=tol)
            assert torch.equal(o1, out[part]) and torch.equal(f1, fell[part])
    smp.close()


# ---- the chi_clamped count of photons that the pair-rate bound lets go ----------------------------------
def _photon_batch(tables, b, kind, flags, steps=3):
    n = len(b["id"])
    bt = Q.Batch(tables, [Q.field(kind, a0=150.0, n_cycles=6.0, phase=2.0, eta0=ETA0)], [3], [(64, 64, n)], 0.2, t0=8.0,
                 flags=flags)
    g = bt.buffers()[0][2]
    g.load(b["pos"], b["mom"], b["spin"], b["w"], b["id"])
    g.init_tau(3)
    bt.step(steps)
    c, q = bt.ctr.read().as_dict(), g.q.cpu().numpy().view(np.uint32)
    c.pop("first_bad")
    bt.close()
    return q, c


@pytest.mark.parametrize("kind", [B.QED_FIELD_LP, B.QED_FIELD_CP])
@pytest.mark.parametrize("chi_max", [0.004, 0.02, 0.1])
def test_pair_rate_bound_counts_clamped_photons(kind, chi_max):
    """Tables that end below the chi at which pair rates begin (0.03): a photon above their end is counted in
    chi_clamped although it has no rate, in the kernels with the bound as in those without."""
    t = Q.Tables(chi_min=1e-3, chi_max=chi_max, n_chi=24, n_r=64)
    b = _photons(20011, 60)
    q0, _, c0 = _pair_steps(t, b, kind, B.QED_F_FULL)
    q1, _, c1 = _pair_steps(t, b, kind, B.QED_F_FULL | B.QED_F_TBMT_PAPER)
    assert c1["chi_clamped"] > 0 and c0 == c1 and np.array_equal(q0, q1)
    for flags in (B.QED_F_FULL, B.QED_F_FULL | B.QED_F_TBMT_PAPER):
        q, c = _photon_batch(t, b, kind, flags)
        assert c["chi_clamped"] == c1["chi_clamped"] and np.array_equal(q, q1)
    t.close()


# ---- the shared-memory limits of kernels that several batches, tables and threads use --------------------
@pytest.mark.parametrize("graph_steps", [0, 2])
def test_live_batches_keep_their_shared_memory(tables, graph_steps):
    """A batch that needs more shared memory than one made or tuned after it (more instances, a longer table) steps
    as it does alone."""
    long_t = Q.Tables(chi_min=1e-3, chi_max=1e2, n_chi=200, n_r=16)

    def make(t, n_inst):
        fields = [Q.field(B.QED_FIELD_CP, a0=150.0, n_cycles=4.0, phase=4 * math.pi, eta0=ETA0)] * n_inst
        bt = Q.Batch(t, fields, list(range(n_inst)), [(200, 200, 2000)] * n_inst, 0.2, t0=1.0)
        bt.set_tuning(graph_steps=graph_steps)
        for k, (e, _, _) in enumerate(bt.buffers()):
            bm = I.lepton_beam(50, 3000.0, z_range=(-3.0, 3.0), seed=k, id_offset=k << 40)
            e.load(bm["pos"], bm["mom"], bm["spin"], bm["w"], bm["id"])
            e.init_tau(k)
        return bt

    def result(bt):
        out = [{k: v[np.argsort(r["id"])] for k, v in r.items()} for trio in bt.buffers() for r in (b.read() for b in trio)]
        st = bt.stats()
        return out, (st.step, st.particle_steps)

    shapes = [(tables, 96), (long_t, 8), (tables, 8)]
    want = []
    for t, n in shapes:
        bt = make(t, n)
        bt.step(4)
        want.append(result(bt))
        bt.close()
    live = [make(t, n) for t, n in shapes]
    for _ in range(2):
        for bt in live:
            bt.step(2)
    for bt, (out, stats) in zip(live, want):
        got, gs = result(bt)
        assert gs == stats
        for a, b in zip(got, out):
            for k in a:
                assert np.array_equal(a[k], b[k]), k
        bt.close()
    long_t.close()


def test_single_buffer_steps_of_two_threads(tables):
    """Threads that step their own particles with tables of different lengths (each on its own stream)."""
    import threading
    long_t = Q.Tables(chi_min=1e-3, chi_max=1e2, n_chi=4000, n_r=8)
    f = Q.field(B.QED_FIELD_CP, a0=50.0, n_cycles=4.0, phase=4 * math.pi, eta0=ETA0)
    failed = []

    def run(t, seed):
        try:
            bm = I.lepton_beam(65, 3000.0, z_range=(-3.0, 3.0), seed=seed)
            e, g, ctr = Q.ParticleBuffer(65, B.QED_FP32, B.QED_ELECTRON), Q.ParticleBuffer(40000, B.QED_FP32, B.QED_PHOTON), Q.Counters()
            e.load(bm["pos"], bm["mom"], bm["spin"], bm["w"], bm["id"])
            e.init_tau(seed)
            stream = torch.cuda.Stream()
            torch.cuda.synchronize()
            for s in range(1500):
                B.qed_push_step(t.handle, f, Q.step_desc(0.01, 0.01 * s, s, seed), e.s, g.s, ctr.ptr, stream.cuda_stream)
            stream.synchronize()
        except Exception as x:  # noqa: BLE001
            failed.append(x)

    threads = [threading.Thread(target=run, args=(t, k)) for k, t in enumerate((tables, long_t, tables, long_t))]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not failed, failed
    torch.cuda.synchronize()
    long_t.close()


# ---- repeatability of the training of small batches ------------------------------------------------------
@pytest.mark.parametrize("n", [1, 64, 128, 129, 300, 640, 1000, 1024])
def test_small_batches_train_bit_for_bit(tables, n):
    """Up to 1024 samples a gradient is summed in a fixed order, so it, its loss and the networks trained on it repeat
    bit for bit."""
    smp = GM.Sampler(GM.init_params(6), max_batch=1024)
    x, y, _ = GM.targets(tables, n, 5, 0)
    g0, l0 = smp.grad(x, y)
    for _ in range(50):
        g, loss = smp.grad(x, y)
        assert torch.equal(g, g0) and torch.equal(loss, l0)
    nets = []
    for _ in range(4):
        smp.set_params(GM.init_params(6))
        loss = smp.train(tables, 12, batch=n, seed=4)
        nets.append((loss, smp.params()))
    for loss, p in nets[1:]:
        assert np.array_equal(loss, nets[0][0]) and np.array_equal(p, nets[0][1])
    smp.close()


# ---- the choice of the plane-wave kernels ---------------------------------------------------------------
@pytest.mark.parametrize("n_chi,n_inst", [(24, 1), (256, 96), (448, 96), (24, 300), (256, 1024), (2048, 8), (4096, 96), (9000, 3)])
def test_plane_wave_kernels_keep_the_blocks_per_sm(n_chi, n_inst):
    """The plane-wave kernels' rate queues cost no variant more than a quarter of the blocks per SM that the kernels
    that read the flags have."""
    t = Q.Tables(chi_min=1e-3, chi_max=1e2, n_chi=n_chi, n_r=4)
    fields = [Q.field(B.QED_FIELD_LP, a0=10.0, n_cycles=4.0, eta0=ETA0)] * n_inst
    got = []
    for flags in (B.QED_F_FULL, B.QED_F_FULL | B.QED_F_TBMT_PAPER):
        bt = Q.Batch(t, fields, [1] * n_inst, [(8, 8, 8)] * n_inst, 0.1, flags=flags)
        per = []
        for v in range(5):
            try:
                bt.set_tuning(variant=v, blocks_per_sm=0, chunk=4, graph_steps=0)
                per.append(bt.tuning().blocks_per_sm)
            except B.QedError:
                per.append(0)
        got.append(per)
        bt.close()
    t.close()
    assert all(4 * a >= 3 * b for a, b in zip(*got)), got


@pytest.mark.parametrize("n_chi", [24, 448, 600, 3000, 6000])
def test_plane_wave_kernels_agree(n_chi):
    """Table lengths on either side of where the rate queues are left out: the photons of a batch are word for word
    those of the kernels that read the flags."""
    t = Q.Tables(chi_min=1e-3, chi_max=1e2, n_chi=n_chi, n_r=8)
    b = _photons(20011, 61)
    got = []
    for flags in (B.QED_F_FULL, B.QED_F_FULL | B.QED_F_TBMT_PAPER):  # (T-BMT concerns leptons only: one step)
        bt = Q.Batch(t, [Q.field(B.QED_FIELD_CP, a0=150.0, n_cycles=6.0, phase=2.0, eta0=ETA0)], [3],
                     [(20011, 20011, 20011)], 0.2, t0=8.0, flags=flags)
        bt.buffers()[0][2].load(b["pos"], b["mom"], b["spin"], b["w"], b["id"])
        bt.buffers()[0][2].init_tau(3)
        bt.step(1)
        c = bt.ctr.read().as_dict()
        c.pop("first_bad")
        got.append(([{k: v[np.argsort(r["id"])] for k, v in r.items()} for r in (x.read() for x in bt.buffers()[0])], c))
        bt.close()
    assert got[0][1] == got[1][1] and got[0][1]["events"] > 0 and got[0][1]["nonfinite"] == 3
    for x, y in zip(got[0][0], got[1][0]):
        for k in x:
            assert np.array_equal(x[k], y[k], equal_nan=True), k
    t.close()


@pytest.mark.parametrize("per_sm", [128, 1024])
@pytest.mark.parametrize("over", [-1, 0, 1, 33])
def test_sampler_at_the_edges_of_its_block_sizes(tables, per_sm, over):
    """The check's blocks have 128 threads up to 128 samples an SM, then 1024, and its tiles are cut so that every
    block takes as many: each sample is what it is in small calls."""
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + over
    chi, r, s = _query(n, 14)
    smp = GM.Sampler(GM.init_params(4))
    for kw in ({}, {"table_only": True}):
        out, fell, nf = smp.sample(tables, chi, r, s, tol=3e-3, **kw)
        assert int(nf) == int(fell.sum()) > 0
        for a in (0, 1000, n // 2, n - 700):
            part = slice(a, min(n, a + 1001))
            o1, f1, _ = smp.sample(tables, chi[part].contiguous(), r[part].contiguous(), s[part].contiguous(), tol=3e-3, **kw)
            assert torch.equal(o1, out[part]) and torch.equal(f1, fell[part])
    smp.close()


def test_mixture_quantile_stays_between_the_branches(tables):
    """s_beta beyond +-1 (a spin of length above 1): the table path's quantile lies between those of the two branches,
    which s_beta = 1 and -1 give."""
    chi, r, _ = _query(20003, 15)
    smp = GM.Sampler(GM.init_params(4))
    at = {s: smp.sample(tables, chi, r, torch.full_like(chi, s), table_only=True)[0][:, 0].double()
          for s in (-4.0, -1.5, -1.0000005, -1.0, 1.0, 1.0000005, 1.2, 3.0)}
    lo, hi = torch.minimum(at[-1.0], at[1.0]), torch.maximum(at[-1.0], at[1.0])
    slack = 1e-8 + 2.0 ** -23 * torch.maximum(lo.abs(), hi.abs())  # one rounding of each float
    for s, got in at.items():
        assert bool(((got >= lo - slack) & (got <= hi + slack)).all()), s
    smp.close()
