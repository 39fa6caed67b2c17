"""What this framework is measured on: the calls its users make, over the sizes they make them at.

A program built on the library (include/qed.h through paper_2511_08929_gb300) builds the rate tables once,
loads beams, and advances them through a laser pulse: either buffer by buffer (qed_push_step, qed_pair_step,
qed_compact, in FP64 or FP32) or many collisions at once (qed_batch_*).  A program that uses the learned
sampler also trains it and draws from it.  Every kind of case below is one of those calls:

  tables   qed_tables_build and the export of everything it built
  single   steps of one collision through the single-buffer entry points, from a state inside the pulse
  batch    a batch created over such states, its steps, its results; `network` draws its emissions
  sample   energy fractions for given (chi, r, s_beta) from the network or from the tables
  train    AdamW steps on fresh table samples

A pass restores the particles of the state (the copy a program makes that runs several configurations from
one checkpoint), advances them and returns every particle.  Daughters are appended in the order the device
reserves their slots, which no two runs share, so the particles come back in the order of their ids, the way
a program that follows particles reads them.  The state is a collision half way through, as the benchmark
times it: the beam inside the pulse, electrons that have radiated, the photons they emitted, some positrons.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2511_08929_gb300 import binding as B
from paper_2511_08929_gb300 import buffers as Q
from paper_2511_08929_gb300 import inputs as I
from paper_2511_08929_gb300 import mlp as M

DT = 2.0 * math.pi / 100.0  # lambda / (100 c), the step of every workload of inputs.py
WAVELENGTH_UM = 0.8
ETA0 = I.eta0_for_wavelength(WAVELENGTH_UM)
BEAM = 20.0 * math.pi  # beam length: ten wavelengths
PHI_FRONT = 51.0  # laser phase of the beam's front end when the pass starts (the pulse covers [0, 20 pi])

FULL = B.QED_F_FULL
FLAGS = {
    "full": FULL,  # the paper's method (the default of every entry point)
    "amm": FULL | B.QED_F_AMM,  # field-dependent anomalous moment in T-BMT (Sec. 8.6.2)
    "loop": FULL | B.QED_F_LOOP,  # the same moment as the one-loop term of the no-emission update (App. A.1)
    "beta": FULL | B.QED_F_BETA_BASIS,  # spins along +-beta (Sec. 8.3)
    "reject": FULL | B.QED_F_REJECT,  # table-free sampling (Sec. 4.2)
    "mean": FULL & ~(B.QED_F_SPIN_COLLAPSE | B.QED_F_POL_COLLAPSE),  # expectation values, no collapse
    "averaged": FULL & ~B.QED_F_RESOLVED,  # spin-averaged rates
    "probability": FULL & ~B.QED_F_TAU,  # per-step probability instead of the optical depth (Sec. 4.1)
}


# ---- the cases -----------------------------------------------------------------------------------------
def listed():
    return [
        # every program starts with this: the tables of all workloads of inputs.py
        {"name": "tables_256x256", "kind": "tables", "n_chi": 256, "n_r": 256},
        # the smallest step calls, where latency and launches count: 1e4 electrons in the linear pulse of the
        # "plain FP64 method, small" workload, emission only, in both arithmetic paths
        {"name": "push_fp64_1e4", "kind": "single", "fp64": True, "pairs": False, "laser": "LP", "a0": 50.0,
         "gamma": 2000.0, "n": 10000, "photons": 4.0, "steps": 32, "flags": "full"},
        {"name": "push_fp32_1e4", "kind": "single", "fp64": False, "pairs": False, "laser": "LP", "a0": 50.0,
         "gamma": 2000.0, "n": 10000, "photons": 4.0, "steps": 64, "flags": "full"},
        # the coupled species of the head-on circular workload, plain FP64 path (odd size)
        {"name": "headon_fp64_1e5", "kind": "single", "fp64": True, "pairs": True, "laser": "CP", "a0": 150.0,
         "gamma": 4000.0, "n": 100003, "photons": 10.0, "steps": 4, "flags": "full"},
        # and its FP32 path at scale
        {"name": "headon_fp32_1e6", "kind": "single", "fp64": False, "pairs": True, "laser": "CP", "a0": 150.0,
         "gamma": 4000.0, "n": 1000000, "photons": 10.0, "steps": 48, "flags": "full"},
        # a handful of small collisions (a quick scan): launches and gaps
        {"name": "batch8_small", "kind": "batch", "inst": 8, "n_min": 500, "n_max": 5000, "photons": 10.0,
         "steps": 256, "flags": "full", "network": False},
        # the 96-collision workload with beams of 1e3 to 2e4 electrons
        {"name": "batch96_mid", "kind": "batch", "inst": 96, "n_min": 1000, "n_max": 20000, "photons": 10.0,
         "steps": 96, "flags": "full", "network": False},
        # the 96-collision workload with beams of up to 5e5 electrons: the benchmark's regime
        {"name": "batch96_large", "kind": "batch", "inst": 96, "n_min": 1000, "n_max": 500000, "photons": 11.0,
         "steps": 96, "flags": "full", "network": False},
        # the two-pulse cascade (one instance, counter-propagating waves, photons above 300 mc^2)
        {"name": "cascade_2e6", "kind": "cascade", "n": 2000003, "steps": 48, "flags": "full"},
        # the learned sampler in the batched step
        {"name": "batch96_network", "kind": "batch", "inst": 96, "n_min": 1000, "n_max": 100000, "photons": 10.0,
         "steps": 48, "flags": "full", "network": True},
        # the learned sampler on its own, a step's worth of events
        {"name": "sample_1e6", "kind": "sample", "n": 1000003, "mode": "network"},
        # and its training at the batch size of the learned-sampler workload
        {"name": "train_4096", "kind": "train", "batch": 4096, "steps": 16},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tables", "single", "single", "single", "batch", "batch", "batch", "cascade", "sample", "train"])
    flags = "full" if rng.random() < 0.6 else rng.choice(sorted(set(FLAGS) - {"full"}))
    if kind == "tables":
        return {"kind": kind, "n_chi": rng.randint(48, 256), "n_r": rng.randint(48, 256)}
    if kind == "single":
        fp64, pairs = rng.random() < 0.4, rng.random() < 0.6
        n = _log_int(rng, 3000, 100000 if fp64 else 1000000)
        return {"kind": kind, "fp64": fp64, "pairs": pairs, "laser": rng.choice(["LP", "CP"]),
                "a0": round(rng.uniform(10.0, 300.0), 2), "gamma": round(rng.uniform(500.0, 8000.0), 1), "n": n,
                "photons": round(rng.uniform(2.0, 10.0), 2), "steps": rng.randint(2, 6) if fp64 else rng.randint(16, 48),
                "flags": flags}
    if kind == "batch":
        inst = _log_int(rng, 1, 128)
        return {"kind": kind, "inst": inst, "n_min": _log_int(rng, 300, 1000),
                "n_max": _log_int(rng, 1500, 200000), "photons": round(rng.uniform(5.0, 11.0), 2),
                "steps": rng.randint(32, 96), "flags": flags,
                "network": flags != "reject" and rng.random() < 0.2}
    if kind == "cascade":
        return {"kind": kind, "n": _log_int(rng, 20000, 2000000), "steps": rng.randint(16, 48), "flags": flags}
    if kind == "sample":
        return {"kind": kind, "n": _log_int(rng, 2000, 2000000),
                "mode": rng.choice(["network", "network", "branch", "quantile"])}
    return {"kind": kind, "batch": _log_int(rng, 500, 8192), "steps": rng.randint(8, 16)}


# ---- what a program keeps: tables, a trained network --------------------------------------------------
_kept = {}


def _tables():
    if "tables" not in _kept:
        _kept["tables"] = Q.Tables(n_chi=256, n_r=256)
    return _kept["tables"]


def _trained():
    """Parameters of a trained network, from Adam steps in torch on table samples: the same in every process,
    whatever the library's own training kernels do."""
    if "net" not in _kept:
        x, y, _ = M.targets(_tables(), 65536, seed=11)
        names = [name for name, _ in M.LAYOUT]
        p = [torch.tensor(M.unflatten(M.init_params(5))[k], dtype=torch.float32, device="cuda", requires_grad=True)
             for k in names]
        opt = torch.optim.Adam(p, lr=torch.tensor(0.0, device="cuda"), capturable=True, foreach=True)
        steps, batch = 6000, 4096
        xb, yb = x[:batch].clone(), y[:batch].clone()

        def update():
            h = xb
            for layer in range(4):
                h = torch.addmm(p[2 * layer + 1], h, p[2 * layer].T)
                h = torch.nn.functional.silu(h) if layer < 3 else h
            opt.zero_grad(set_to_none=False)
            (h - yb).square().sum(1).mean().backward()
            opt.step()

        side, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            for _ in range(3):  # at learning rate 0: makes the gradients and the optimiser's state
                update()
        torch.cuda.current_stream().wait_stream(side)
        with torch.cuda.graph(graph):
            update()
        for k in range(steps):
            a = (k % (len(x) // batch)) * batch
            xb.copy_(x[a:a + batch])
            yb.copy_(y[a:a + batch])
            opt.param_groups[0]["lr"].fill_(1e-5 + 4e-3 * 0.5 * (1.0 + math.cos(math.pi * k / steps)))
            graph.replay()
        _kept["net"] = M.flatten({k: v.detach().cpu().numpy() for k, v in zip(names, p)})
    return _kept["net"]


# ---- particles inside a pulse -------------------------------------------------------------------------
def _unit(gen, n):
    v = torch.randn((n, 3), generator=gen, device="cuda")
    return v / v.norm(dim=1, keepdim=True)


def _norm(v):
    return v / v.norm(dim=1, keepdim=True).clamp_min(1e-30)


def _per(insts, counts, key):
    v = torch.tensor([float(i[key]) for i in insts], device="cuda")
    return torch.repeat_interleave(v, torch.tensor(counts, device="cuda"))


def _ids(counts, species):
    out = [torch.arange(c, device="cuda") + ((k << 40) + (species << 37) + 1) for k, c in enumerate(counts)]
    return torch.cat(out)


def _pulse_leptons(gen, insts, counts, species):
    """Leptons of every collision, one after the other: spread over the beam, along -z with the transverse
    momentum the wave gives them, energies down to a fifth of the beam's (they have radiated)."""
    n = sum(counts)
    rand = lambda: torch.rand(n, generator=gen, device="cuda")  # noqa: E731
    a0, g0, cp = _per(insts, counts, "a0"), _per(insts, counts, "gamma"), _per(insts, counts, "cp")
    z = BEAM * rand()
    phi = PHI_FRONT - z
    a = torch.where(phi > 0, a0 * torch.sin(phi / 20.0) ** 2, torch.zeros_like(phi))
    px, py = a * torch.sin(phi), -cp * a * torch.cos(phi)
    gam = g0 * torch.exp(-1.6 * rand() * (0.3 if species == 0 else 1.0)) * (1.0 if species == 0 else 0.3) + 30.0
    pz = -torch.sqrt((gam * gam - 1.0 - px * px - py * py).clamp_min(1.0))
    pos = torch.stack([torch.zeros_like(z), torch.zeros_like(z), z], 1)
    return pos, torch.stack([px, py, pz], 1), _unit(gen, n), _ids(counts, species)


def _pulse_photons(gen, insts, counts):
    """The photons such leptons have emitted: the synchrotron spectrum (u' falls as u'^-2/3 e^-u'), along the
    emitter's momentum, polarized along the wave's electric field at the emission."""
    n = sum(counts)
    rand = lambda: torch.rand(n, generator=gen, device="cuda")  # noqa: E731
    a0, g0, cp = _per(insts, counts, "a0"), _per(insts, counts, "gamma"), _per(insts, counts, "cp")
    psi = 2.0 * math.pi * rand()
    a = a0 * torch.sin(math.pi * rand()) ** 2
    gam = g0 * torch.exp(-1.6 * rand())
    tx, ty = a * torch.sin(psi) / gam, -cp * a * torch.cos(psi) / gam
    chi = (2.0 * ETA0 * gam * a).clamp_min(1e-4)
    up = rand() ** 3 * (-torch.log(rand().clamp_min(1e-12))) ** 0.8
    k = gam * (3.0 * chi * up / (2.0 + 3.0 * chi * up)).clamp_min(1e-12)
    k = torch.minimum(k, 0.5 / (ETA0 * a0))  # harder ones have made pairs
    d = _norm(torch.stack([tx, ty, -torch.ones_like(tx)], 1))
    e = torch.stack([torch.where(cp > 0, torch.cos(psi), torch.ones_like(psi)), cp * torch.sin(psi),
                     torch.zeros_like(psi)], 1)
    P = _norm(e - (e * d).sum(1, keepdim=True) * d)
    z = BEAM * rand()
    pos = torch.stack([torch.zeros_like(z), torch.zeros_like(z), z], 1)
    return pos, k[:, None] * d, P, _ids(counts, 2)


def _cascade_particles(gen, counts):
    """Leptons and photons where two circular pulses overlap: momenta mostly across the laser axis, photons
    above the storage threshold."""
    out = []
    for species, n in enumerate(counts):
        rand = lambda: torch.rand(n, generator=gen, device="cuda")  # noqa: B023,E731
        ph, up = 2.0 * math.pi * rand(), torch.randn(n, generator=gen, device="cuda") * 0.5
        d = _norm(torch.stack([torch.cos(ph), torch.sin(ph), up], 1))
        en = 300.0 - 250.0 * torch.log(rand().clamp_min(1e-9)) if species == 2 else 100.0 + 900.0 * rand()
        z = (rand() - 0.5) * 4.0 * math.pi
        pos = torch.stack([torch.zeros_like(z), torch.zeros_like(z), z], 1)
        s = _unit(gen, n)
        if species == 2:
            s = _norm(s - (s * d).sum(1, keepdim=True) * d)
        out.append((pos, en[:, None] * d, s, _ids([n], species)))
    return out


def _fill(buf, pos, mom, spin, ids, seed):
    """Particles on the device into a buffer's planes (the layouts of qed.h), weights 1, optical depths drawn."""
    n = len(ids)
    if buf.layout == B.QED_FP64:
        for i, v in enumerate((pos, mom, spin)):
            buf.planes[3 * i:3 * i + 3, :n] = v.T.double()
        buf.planes[10, :n] = 1.0
    elif buf.charge == B.QED_PHOTON:
        buf.q[0, :n, 0:3], buf.q[0, :n, 3], buf.q[1, :n, 0:2] = pos, spin[:, 0], spin[:, 1:3]
        buf.q[2, :n, 0:3], buf.q[2, :n, 3] = mom, 1.0
    else:
        buf.q[0, :n, 0:3], buf.q[0, :n, 3], buf.q[1, :n, 0:2] = pos, mom[:, 0], mom[:, 1:3]
        buf.q[1, :n, 2:4], buf.q[2, :n, 0], buf.q[2, :n, 1] = spin[:, 0:2], spin[:, 2], 1.0
    buf.ids[:n] = ids
    buf.counts.fill_(n)
    buf.init_tau(seed)


class _State:
    """Buffers per collision (electrons, positrons, photons) with a copy of what they hold."""

    def __init__(self, bufs):
        self.bufs = bufs  # [(e, p, g)]
        flat = [b for t in bufs for b in t]
        self.live, self.saved, self.live_i, self.saved_i = [], [], [], []
        for b in flat:
            n = b.count()
            planes = [b.planes[i, :n] for i in range(11)] if b.layout == B.QED_FP64 else [b.q[i, :n] for i in range(3)]
            if n:
                self.live += planes
                self.live_i.append(b.ids[:n])
            self.live_i.append(b.counts)
            if hasattr(b, "n_dead"):
                self.live_i.append(b.n_dead)
        self.saved = [t.clone() for t in self.live]
        self.saved_i = [t.clone() for t in self.live_i]
        self.ctr = Q.Counters()

    def restore(self):
        torch._foreach_copy_(self.live, self.saved)
        torch._foreach_copy_(self.live_i, self.saved_i)
        self.ctr.zero()

    def results(self):
        """Every particle of every collision, by species and in the order of the ids, and the counters.  The
        arrays are as long as the buffers together; what lies beyond the particles alive is zero."""
        counts = torch.stack([b.counts[0] for t in self.bufs for b in t]).cpu().tolist()
        c = self.ctr.read()
        out = {"events": c.events, "stored": c.stored, "dropped": c.dropped_capacity, "nonfinite": c.nonfinite}
        for sp, name in enumerate(("electrons", "positrons", "photons")):
            bs = [(t[sp], counts[3 * k + sp]) for k, t in enumerate(self.bufs)]
            room, n = sum(b.capacity for b, _ in bs), sum(m for _, m in bs)
            if not room:
                continue
            ids = torch.zeros(room, dtype=torch.int64, device="cuda")
            ids[:n], order = torch.sort(torch.cat([b.ids[:m] for b, m in bs]))
            if bs[0][0].layout == B.QED_FP64:
                v = torch.zeros((11, room), dtype=torch.float64, device="cuda")
                v[:, :n] = torch.cat([b.planes[:, :m] for b, m in bs], 1)[:, order]
                got = {"pos": v[0:3], "mom": v[3:6], "spin": v[6:9], "tau": v[9], "w": v[10]}
            else:
                q0, q1, q2 = (torch.empty((room, 4), device="cuda") for _ in range(3))
                for i, q in enumerate((q0, q1, q2)):
                    q[n:] = 0.0
                    rows = torch.cat([b.q[i, :m] for b, m in bs]).view(torch.complex128)[:, 0]  # 16 bytes each
                    torch.index_select(rows, 0, order, out=q[:n].view(torch.complex128)[:, 0])
                if sp == 2:
                    got = {"P_x": q0[:, 3], "P_yz": q1[:, 0:2], "k": q2[:, 0:3], "w": q2[:, 3]}
                    tau = q1[:, 2:4]
                else:
                    got = {"p_x": q0[:, 3], "p_yz": q1[:, 0:2], "s_xy": q1[:, 2:4], "s_z": q2[:, 0], "w": q2[:, 1]}
                    tau = q2[:, 2:4]
                got["pos"] = q0[:, 0:3]
                # two words of an FP64 sum of FP32 rates: as accurate as those
                got["tau"] = tau.contiguous().view(torch.float64)[:, 0].float()
            out[name] = {"id": ids, **got}
        return out


def _emitted(a0, steps):
    """An upper estimate of the photons a lepton of these beams emits in so many steps: 5 alpha a0 / (2 sqrt 3)
    a radian of the phase, half of it in the mean over the pulse."""
    return 0.5 * 0.0105 * a0 * 2.0 * DT * steps


def _species_counts(n, photons, pairs=True):
    return n, (n // 7 if pairs else 0), int(n * photons)


def _instances(case):
    if case["kind"] == "batch":
        insts = I.batched_instances(case["inst"], 3, case["n_min"], case["n_max"])
    else:
        insts = [{"n": case["n"], "a0": case["a0"], "gamma": case["gamma"], "kind": case["laser"]}]
    for i in insts:
        i["cp"] = 1.0 if i["kind"] == "CP" else 0.0
    return insts


def _field(inst):
    # phase: the beam's front is at PHI_FRONT at time 0
    kind = B.QED_FIELD_CP if inst["kind"] == "CP" else B.QED_FIELD_LP
    return Q.field(kind, a0=inst["a0"], n_cycles=10.0, phase=PHI_FRONT, eta0=ETA0)


def _collisions(case, gen, seed, layout, pairs):
    insts = _instances(case)
    cnt = list(zip(*[_species_counts(i["n"], case["photons"], pairs) for i in insts]))
    sets = [_pulse_leptons(gen, insts, list(cnt[0]), 0), _pulse_leptons(gen, insts, list(cnt[1]), 1),
            _pulse_photons(gen, insts, list(cnt[2]))]
    bufs, at = [], [0, 0, 0]
    for k, inst in enumerate(insts):
        ne, npos, ng = cnt[0][k], cnt[1][k], cnt[2][k]
        room = int(6e-6 * inst["a0"] * case["steps"] * ng) + 300 if pairs else 0
        caps = (ne + room, npos + room, ng + int((ne + npos + room) * (_emitted(inst["a0"], case["steps"]) + 0.1)) + 1000)
        trio = []
        for sp, charge in enumerate((B.QED_ELECTRON, B.QED_POSITRON, B.QED_PHOTON)):
            n = (ne, npos, ng)[sp]
            b = Q.ParticleBuffer(caps[sp], layout, charge, photons=sp == 2, use_begin=case["kind"] == "single")
            _fill(b, *(v[at[sp]:at[sp] + n] for v in sets[sp]), seed + k)
            at[sp] += n
            trio.append(b)
        bufs.append(tuple(trio))
    return insts, _State(bufs)


def _batch_instances(st, fields, seed):
    out = []
    for k, (trio, f) in enumerate(zip(st.bufs, fields)):
        i = B.QedInstance()
        i.field, i.seed = f, seed + k
        i.electrons, i.positrons, i.photons = (b.s for b in trio)
        out.append(i)
    return out


def _batch_desc(case, t0=0.0, store_min=0.0):
    d = B.QedBatchDesc()
    d.dt, d.t0, d.step0, d.flags, d.photon_store_min = DT, t0, 0, FLAGS[case["flags"]], store_min
    return d


# ---- the contract -------------------------------------------------------------------------------------
def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    kind = case["kind"]
    s = {"case": case, "seed": int(seed)}
    if kind == "tables":
        # the lower end of the grid follows the seed: a program's range follows its laser
        s["chi_min"] = 1e-4 * (1.0 + (int(seed) % 9973) / 9973.0)
        return s
    s["tables"] = _tables()
    if kind == "sample":
        n = case["n"]
        rand = lambda: torch.rand(n, generator=gen, device="cuda", dtype=torch.float64)  # noqa: E731
        s["chi"] = torch.exp(math.log(1e-3) + rand() * math.log(1e5))
        s["r"], s["s"] = rand().clamp(1e-12, 1.0 - 1e-12), 2.0 * rand() - 1.0
        s["sampler"] = M.Sampler(_trained())
    elif kind == "train":
        s["init"] = M.init_params(int(seed))
        s["sampler"] = M.Sampler(s["init"], max_batch=case["batch"])
    elif kind == "single":
        layout = B.QED_FP64 if case["fp64"] else B.QED_FP32
        insts, s["st"] = _collisions(case, gen, s["seed"], layout, case["pairs"])
        s["field"] = _field(insts[0])
        s["ws"] = Q.CompactWorkspace(s["st"].bufs[0][2].capacity)
        s["steps"] = [Q.step_desc(DT, k * DT, k, s["seed"], flags=FLAGS[case["flags"]]) for k in range(case["steps"])]
    elif kind == "batch":
        insts, s["st"] = _collisions(case, gen, s["seed"], B.QED_FP32, True)
        s["insts"], s["desc"] = _batch_instances(s["st"], [_field(i) for i in insts], s["seed"]), _batch_desc(case)
        if case["network"]:
            s["sampler"] = M.Sampler(_trained())
    elif kind == "cascade":
        n = case["n"]
        counts, c = (n, n // 3, n), I.CASCADE_2E8
        k = case["steps"]
        caps = (n + int(0.008 * k * n) + 1000, n // 3 + int(0.008 * k * n) + 1000, n + int(0.04 * k * n) + 1000)
        trio = []
        for sp, (charge, got) in enumerate(zip((B.QED_ELECTRON, B.QED_POSITRON, B.QED_PHOTON),
                                               _cascade_particles(gen, counts))):
            b = Q.ParticleBuffer(caps[sp], B.QED_FP32, charge, photons=sp == 2)
            _fill(b, *got, s["seed"])
            trio.append(b)
        s["st"] = _State([tuple(trio)])
        f = Q.laser_field(c.laser())
        # half way through the two pulses
        s["insts"] = _batch_instances(s["st"], [f], s["seed"])
        s["desc"] = _batch_desc(case, t0=math.pi * c.n_cycles, store_min=c.photon_store_min)
    return s


def _run_tables(s):
    c = s["case"]
    t = Q.Tables(chi_min=s["chi_min"], n_chi=c["n_chi"], n_r=c["n_r"])
    out = t.export()
    out["amm"] = B.qed_tables_export_amm(t.handle, t.desc)
    t.close()
    return out


def _run_single(s):
    st, h = s["st"], s["tables"].handle
    e, p, g = st.bufs[0]
    st.restore()
    pairs = s["case"]["pairs"]
    for d in s["steps"]:
        if pairs:
            B.qed_snapshot_counts([e.s, p.s, g.s])
            B.qed_pair_step(h, s["field"], d, g.s, e.s, p.s, st.ctr.ptr)
            B.qed_push_step(h, s["field"], d, e.s, g.s, st.ctr.ptr)
            B.qed_push_step(h, s["field"], d, p.s, g.s, st.ctr.ptr)
            B.qed_compact(g.s, s["ws"].ptr, s["ws"].bytes)
        else:
            B.qed_snapshot_counts([e.s])
            B.qed_push_step(h, s["field"], d, e.s, g.s, st.ctr.ptr)
    return st.results()


def _run_batch(s):
    st = s["st"]
    st.restore()
    h = B.qed_batch_create(s["tables"].handle, s["insts"], s["desc"], st.ctr.ptr)
    if "sampler" in s:
        B.qed_batch_set_mlp(h, s["sampler"].handle, 1e-4)
    B.qed_batch_step(h, s["case"]["steps"])
    out = st.results()
    B.qed_batch_destroy(h)
    return out


def run(s):
    kind = s["case"]["kind"]
    if kind == "tables":
        return _run_tables(s)
    if kind == "single":
        return _run_single(s)
    if kind in ("batch", "cascade"):
        return _run_batch(s)
    if kind == "sample":
        mode = s["case"]["mode"]
        out, fell, nf = s["sampler"].sample(s["tables"], s["chi"], s["r"], s["s"], table_only=mode == "quantile",
                                            branch_table=mode == "branch")
        return {"out": out, "fell": fell, "fallbacks": nf}
    smp = s["sampler"]
    smp.set_params(s["init"])
    loss = smp.train(s["tables"], s["case"]["steps"], batch=s["case"]["batch"], seed=s["seed"])
    return {"loss": loss, "params": smp.params()}


def work(case):
    """Bytes: what the calls have to move.  A step reads and writes every particle once (FP32: x, p, s, tau of a
    lepton 44 + 44; x, k, P, tau of a photon 44 and its position 12, its P and tau 20 more where it can make a
    pair, about a third of them; FP64: twice that).  Operations: a lepton's push, precession, basis, rates and
    update about 400, a photon's move, chi and rates about 150; of a table entry the quadratures that find it."""
    kind = case["kind"]
    if kind == "tables":
        n, m = 4 * case["n_chi"] * case["n_r"], 4 * case["n_chi"]
        return {"bytes": 8.0 * (n + m), "flops": n * 13.0 * 100.0 * 3.0}
    if kind == "sample":
        n = case["n"]
        return {"bytes": n * 41.0, "flops": n * (2.0 * 8640 if case["mode"] == "network" else 300.0)}
    if kind == "train":
        n = case["batch"] * case["steps"]
        return {"bytes": case["steps"] * 4.0 * 7 * B.QED_MLP_PARAMS, "flops": n * 6.0 * 8640}
    if kind == "cascade":
        lep, ph, b, share = case["n"] * 4 // 3, case["n"], 1.0, 1.0
    else:
        c = [_species_counts(i["n"], case["photons"], kind == "batch" or case["pairs"]) for i in _instances(case)]
        lep, ph = sum(x[0] + x[1] for x in c), sum(x[2] for x in c)
        if kind == "single" and not case["pairs"]:
            ph = 0
        b, share = 2.0 if case.get("fp64") else 1.0, 0.3
    return {"bytes": case["steps"] * b * (88.0 * lep + (56.0 + 20.0 * share) * ph),
            "flops": case["steps"] * (400.0 * lep + 150.0 * ph)}


# ---- 64-bit answers -----------------------------------------------------------------------------------
# The tables are integrals: they are taken here by quadrature in torch, in FP64.  Steps, samples and training
# draw events and then branch on them: a 64-bit answer for those would be a second implementation of the
# whole method, so they have none here and are held to the bounds of their types.
def _bessel(x):
    """e^x (K_1/3, K_2/3, int_x^inf K_1/3) by the trapezoid rule on their integrals over cosh (DLMF 10.32.9)."""
    h = torch.clamp(0.6 / torch.sqrt(x), max=0.2)
    end = torch.acosh(1.0 + (46.0 + (2.0 / 3.0) * torch.acosh(1.0 + 46.0 / x)) / x)
    out = [torch.full_like(x, 0.5) for _ in range(3)]
    for m in range(1, int(torch.ceil((end / h).max()).item()) + 1):
        t = m * h
        e = torch.where(t <= end + h, torch.exp(-2.0 * x * torch.sinh(0.5 * t) ** 2), torch.zeros_like(t))
        c = torch.cosh(t / 3.0)
        out[0] += e * c
        out[1] += e * (2.0 * c * c - 1.0)
        out[2] += e * c / torch.cosh(t)
    return [o * h for o in out]


def _density(nbw, chi, sigma, t):
    """Density in t of the spectrum (NLC: u' = t^3; NBW, folded about 1/2: u~' = 8/(3 chi) + t^2)."""
    if nbw:
        u = 8.0 / (3.0 * chi) + t * t
        k13, k23, ik = _bessel(u)
        return (ik + (1.5 * chi * u - 2.0 - sigma) * k23) * torch.exp(-t * t) * 4.0 / (3.0 * chi * u * torch.sqrt(u))
    u = t ** 3
    k13, k23, ik = _bessel(u.clamp_min(1e-60))
    den = 2.0 + 3.0 * chi * u
    lam, om = 3.0 * chi * u / den, 2.0 / den
    return torch.exp(-u) * (-ik + (1.0 / om + om) * k23 + sigma * lam * k13) * 18.0 * chi / (den * den) * t * t


def _exact_tables(case, seed):
    n_chi, n_r, chi_min, chi_max = case["n_chi"], case["n_r"], prepare(case, seed)["chi_min"], 1e3
    D = dict(dtype=torch.float64, device="cuda")
    lnchi = math.log(chi_min) + torch.arange(n_chi, **D) * ((math.log(chi_max) - math.log(chi_min)) / (n_chi - 1))
    chi = torch.exp(lnchi)
    gx, gw = (torch.tensor(v, **D) for v in np.polynomial.legendre.leggauss(12))
    r = torch.sigmoid(-20.0 + 40.0 * torch.arange(n_r, **D) / (n_r - 1))
    out = {"nlc_rate": torch.zeros(2, n_chi, **D), "nbw_rate": torch.zeros(2, n_chi, **D),
           "nlc_icdf": torch.zeros(2, n_chi, n_r, **D), "nbw_icdf": torch.zeros(2, n_chi, n_r, **D)}
    for nbw in (False, True):
        end = math.sqrt(80.0) if nbw else 80.0 ** (1.0 / 3.0)
        edges = torch.linspace(0.0, end, int(16 * end) + 2, **D)
        mid, half = 0.5 * (edges[1:] + edges[:-1]), 0.5 * (edges[1:] - edges[:-1])
        nodes = mid[:, None] + half[:, None] * gx
        for s, sigma in enumerate((1.0, -1.0)):
            c = chi[:, None, None]
            part = (_density(nbw, c, sigma, nodes[None]) * gw).sum(2) * half
            cum = torch.cat([torch.zeros(n_chi, 1, **D), part.cumsum(1)], 1)
            total = cum[:, -1:]
            out["nbw_rate" if nbw else "nlc_rate"][s] = torch.log((2.0 if nbw else 1.0) * total[:, 0])
            want = r[None] * total
            p = (torch.searchsorted(cum, want, right=True) - 1).clamp(0, len(mid) - 1)
            a, below = edges[p], cum.gather(1, p)
            t = a + (edges[p + 1] - a) * (want - below) / (cum.gather(1, p + 1) - below)
            lo, hi = a.clone(), edges[p + 1].clone()
            for _ in range(12):
                m, w = 0.5 * (a + t)[..., None], 0.5 * (t - a)
                F = below + (_density(nbw, c, sigma, m + w[..., None] * gx) * gw).sum(2) * w - want
                lo, hi = torch.where(F > 0, lo, t), torch.where(F > 0, t, hi)
                tn = t - F / _density(nbw, chi[:, None], sigma, t)
                found = (tn - t).abs() <= 1e-14 * t
                t = torch.where(found | ((tn > lo) & (tn < hi)), tn, 0.5 * (lo + hi))
                if bool(found.all()):
                    break
            out["nbw_icdf" if nbw else "nlc_icdf"][s] = (2.0 if nbw else 3.0) * torch.log(t)
    # a(chi) = (alpha/chi) int dv u^2/(1+u)^3 Gi(z)/sqrt z, u = chi e^v, sqrt z = e^(v/3): Gi, from its integral
    # along the ray e^(i pi/6), is needed at the same v for every chi
    lo, hi = -21.0 - max(float(lnchi[-1]), 0.0), 21.0 + max(-float(lnchi[0]), 0.0)
    edges = torch.linspace(lo, hi, int(4 * (hi - lo)) + 1, **D)
    v = (0.5 * (edges[1:] + edges[:-1]))[:, None] + 0.5 * (edges[1] - edges[0]) * gx
    z = torch.exp(2.0 * v / 3.0)
    S = torch.clamp(92.0 / z, max=5.2)[..., None, None]
    ray = (torch.arange(40, **D)[:, None] + 0.5 + 0.5 * gx) / 40.0 * S
    gi = (torch.exp(-ray ** 3 / 3.0 - 0.5 * z[..., None, None] * ray)
          * torch.sin(math.sqrt(0.75) * z[..., None, None] * ray + math.pi / 6.0) * gw).sum((2, 3)) * S[..., 0, 0] / 80.0
    u = chi[:, None, None] * torch.exp(v)
    a = ((u / (1.0 + u)) ** 2 / (1.0 + u) * gi / math.pi * torch.exp(-v / 3.0) * gw).sum((1, 2))
    out["amm"] = torch.log(7.2973525693e-3 / chi * a * 0.5 * (edges[1] - edges[0]))
    return {k: x.cpu().numpy() for k, x in out.items()}


def exact(case, seed):
    return _exact_tables(case, seed) if case["kind"] == "tables" else None
