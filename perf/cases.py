"""What a user of the scheduler has it do, as measurable cases.

Every case is one kind of program around a ``Scheduler`` at one size:

    loop        the scheduler's life: one new loss per running job from host arrays, then one epoch into a
                host array (``append_losses`` + ``schedule``)
    device      the same loop for trainers that leave their losses on the GPU (``append_losses_device`` +
                ``schedule_device``)
    epoch       one epoch over stored histories, result on the GPU (``schedule_device``)
    restart     a scheduler takes over a running cluster: bulk load of all histories, time laws, first epoch
    predict     an epoch and the read-back of everything it predicted, gain rows included
    checkpoint  the state of one scheduler carried into another one, which then schedules
    sharded     one cluster whose jobs are split over several handles, exchanged step by step
    allocate    the allocation step alone on a device table of gains (``allocate_static``)

Jobs are the two convergence families of the benchmark's generators with the same parameter ranges, noise and
iteration-time laws; histories are drawn on the GPU from the seed and handed over as the arrays a program holds.
"""

from __future__ import annotations

import math

import numpy as np
import torch

import paper_1802_04819_b200 as slaq
from paper_1802_04819_b200 import binding as B

# Algorithmic fp64 operations of the fit per stored loss: one sweep of each family, and the set-up
# (normalisation, first guesses).
FLOP_SWEEPS, FLOP_SETUP = 65.0, 40.0
FLOP_GAIN = 30.0


def _case(name, kind, jobs, hist, cap, cores_per_job, **more):
    case = dict(
        kind=kind, jobs=jobs, hist=hist, cap=cap, cores_per_job=float(cores_per_job), epoch_s=3.0,
        packed=False,      # histories kept packed as loaded (each window keeps its length) instead of rings
        stages=False,      # full rings in three stages (new / in training / converged) instead of ragged windows
        law="fixed",       # iteration-time laws: given, or estimated from the reported times ("samples")
        warm=False,        # refits start from the last epoch's curves and take 5 trials instead of 20
        pinned=False,      # the host arrays are page-locked
        selection=0,       # SLAQ_P_SELECTION
        options=False,     # concave envelope and target-loss hints on
        shards=1,
    )
    case.update(more)
    if name is not None:
        case["name"] = name
    return case


def listed():
    return [
        # The smallest cluster of the configurations, in its loop: launches and latency are all there is.
        _case("loop 8 jobs", "loop", 8, 20, 16, 8, law="samples"),
        # The size of the published cluster experiment (160 jobs on 640 cores), reporting iteration times.
        _case("loop 160 jobs", "loop", 160, 40, 32, 4, law="samples"),
        # The published scalability experiment (4,000 jobs on 16,000 cores), losses from ordinary host arrays.
        _case("loop 4000 jobs", "loop", 4000, 200, 64, 4),
        # A large cluster refitting every epoch from the curves of the last one: the production loop.
        _case("loop 100000 jobs warm", "loop", 100_000, 1000, 64, 4, epoch_s=1.0, packed=True, warm=True, pinned=True),
        # Trainers on the same GPU: nothing passes through the host.
        _case("device loop 33000 jobs", "device", 33_000, 128, 64, 4),
        # The benchmark's headline: ragged histories of up to 1,000 losses, every job fitted from its first guess.
        _case("epoch 100000 jobs", "epoch", 100_000, 1000, 64, 4, epoch_s=1.0, packed=True),
        # The largest configuration: a million full rings, 128 cores per job at most, tied jobs among them.
        _case("epoch 1000000 jobs", "epoch", 1_000_000, 64, 128, 4, epoch_s=1.0, stages=True),
        # A scheduler process takes over a cluster in the middle of its life.
        _case("restart 20000 jobs", "restart", 20_000, 200, 64, 4),
        # An operator looks at everything that was predicted, with both prediction options in use.
        _case("predict 4000 jobs", "predict", 4000, 200, 64, 4, options=True),
        # A checkpoint is written and another scheduler continues from it.
        _case("checkpoint 10000 jobs", "checkpoint", 10_000, 64, 64, 4, law="samples"),
        # One cluster in two shards: the multi-GPU protocol.
        _case("sharded 2 x 10000 jobs", "sharded", 20_000, 100, 64, 4, shards=2),
        # A plug-in that must not allocate: the selection alone on a table of gains.
        _case("allocate 20000 rows", "allocate", 20_000, 0, 64, 4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the kinds in turn by chance, sizes over their whole range, every option now and then."""
    kind = rng.choice(["loop", "loop", "loop", "device", "epoch", "epoch", "restart", "predict", "checkpoint",
                       "sharded", "allocate"])
    most = {"loop": 100_000, "device": 100_000, "epoch": 1_000_000, "restart": 40_000, "predict": 20_000,
            "checkpoint": 20_000, "sharded": 60_000, "allocate": slaq.STATIC_MAX_JOBS}[kind]
    jobs = _log_int(rng, 8, most)
    hist = min(_log_int(rng, 8, 1000), max(8, 30_000_000 // jobs))
    cap = _log_int(rng, 4, 128)
    if kind == "allocate":
        return _case(None, kind, jobs, 0, cap, math.exp(rng.uniform(math.log(0.5), math.log(cap))))
    shards = rng.choice([2, 3, 4]) if kind == "sharded" else 1
    plain = kind in ("loop", "device", "epoch", "restart")
    return _case(
        None, kind, jobs, hist, cap, math.exp(rng.uniform(math.log(0.5), math.log(max(1.0, cap / 2)))),
        epoch_s=rng.choice([1.0, 3.0]), packed=kind in ("loop", "epoch", "restart", "sharded") and rng.random() < 0.4,
        stages=rng.random() < 0.25, law=rng.choice(["fixed", "samples"]) if kind in ("loop", "checkpoint") else "fixed",
        warm=kind in ("loop", "device") and rng.random() < 0.4, pinned=kind in ("loop", "restart") and rng.random() < 0.4,
        selection=1 if plain and rng.random() < 0.15 else 0, options=kind in ("epoch", "predict") and rng.random() < 0.4,
        shards=shards)


# ---- inputs ----

def _host(t, pinned=False):
    """A device tensor as the host array a program would hold."""
    return t.cpu().pin_memory().numpy() if pinned else t.cpu().numpy()


class _Jobs:
    """Curves, time laws and stored windows of a cluster, on the GPU."""

    def __init__(self, case, seed):
        g = torch.Generator(device="cuda").manual_seed(seed)
        n, hmax = case["jobs"], case["hist"]
        self.g, self.n = g, n
        u = lambda lo, hi: lo + (hi - lo) * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)   # noqa: E731
        self.expo = u(0, 1) < 0.5
        self.sub_p = (u(1e-4, 1e-2), u(0.01, 1.0), u(0.5, 2.0), u(0.0, 0.1))
        self.exp_p = (u(0.80, 0.99), u(0.0, 5.0), u(0.0, 0.1))
        self.s, self.w = u(0.05, 0.5), torch.exp(u(0.0, math.log(1000.0)))
        H = torch.randint(3, hmax + 1, (n,), generator=g, device="cuda")
        stage, far = u(0, 1), torch.randint(0, 501, (n,), generator=g, device="cuda")
        zero = torch.zeros_like(far)
        if case["stages"]:
            # 20 % new jobs of a few points, 60 % in training, 20 % converged; the windows are full
            H = torch.where(stage < 0.2, 3 + far % 3, torch.full_like(H, hmax))
            self.k0 = torch.where(stage < 0.2, zero, torch.where(stage < 0.8, far, zero + 10_000))
        else:
            self.k0 = torch.where(stage < 0.9, zero, zero + 10_000)   # one job in ten has converged
        self.H, self.sigma = H, torch.full((n,), 0.01, device="cuda", dtype=torch.float64)
        past = torch.full((n,), -math.inf, device="cuda", dtype=torch.float64)
        every = torch.arange(n, device="cuda")
        for k in range(1, 121):   # both families' steepest step lies among the first hundred or so
            step = self.curve(every, self.k0 * 0 + (k - 1)) - self.curve(every, self.k0 * 0 + k)
            past = torch.where(self.k0 >= k, torch.maximum(past, step), past)
        done = self.k0 >= 10_000
        if case["stages"]:
            # a converged job's noise is far below the reductions of its earlier life
            quiet = 1e-4 * past / (self.curve(every, self.k0) * 7.1)
            self.sigma = torch.where(done, torch.minimum(self.sigma, quiet), self.sigma)
        self.offsets = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
        torch.cumsum(H, 0, out=self.offsets[1:])
        total = int(self.offsets[-1])
        owner = torch.repeat_interleave(every, H)
        pos = torch.arange(total, device="cuda") - self.offsets[:-1][owner]
        self.losses = self.noisy(owner, self.k0[owner] + pos)
        if case["stages"] and n >= 200:   # one job in a hundred is an exact copy of another: tied gains
            full = torch.nonzero(H == hmax).flatten()
            pick = full[torch.randperm(full.numel(), generator=g, device="cuda")[: 2 * (n // 100)]]
            src, dst = pick[: pick.numel() // 2], pick[pick.numel() // 2:][: pick.numel() // 2]
            along = torch.arange(hmax, device="cuda")[None, :]
            self.losses[self.offsets[dst][:, None] + along] = self.losses[self.offsets[src][:, None] + along]
            for v in (self.s, self.w, self.k0, past, self.sigma, self.expo, *self.sub_p, *self.exp_p):
                v[dst] = v[src]
        self.m_past, self.k_last = past, self.k0 + H - 1

    def curve(self, j, k):
        k = k.double()
        a, b, c, d = (p[j] for p in self.sub_p)
        mu, b0, c0 = (p[j] for p in self.exp_p)
        return torch.where(self.expo[j], torch.pow(mu, k - b0) + c0, 1.0 / ((a * k + b) * k + c) + d)

    def noisy(self, j, k):
        z = torch.randn(j.numel(), generator=self.g, device="cuda", dtype=torch.float64)
        return self.curve(j, k) * torch.exp(self.sigma[j] * z)


def _scheduler(case, n):
    s = slaq.Scheduler(n, case["hist"], case["cap"])
    if case["warm"]:
        s.set_param(B.P_WARM_START, 1)
        s.set_param(B.P_LM_TRIALS, 5)
    if case["selection"]:
        s.set_param(B.P_SELECTION, case["selection"])
    if case["options"]:
        s.set_param(B.P_GAIN_ENVELOPE, 1)
    return s


def _samples(j, cores):
    return j.s + j.w / cores


def prepare(case, seed):
    kind, n = case["kind"], case["jobs"]
    cores = int(round(case["cores_per_job"] * n))
    st = dict(kind=kind, T=case["epoch_s"], C=cores, at=0)
    if kind == "allocate":
        # gain rows as an epoch's prediction leaves them: falling, over many orders of magnitude between jobs, a
        # tenth of the jobs predicting nothing
        g = torch.Generator(device="cuda").manual_seed(seed)
        u = lambda: torch.rand(n, 1, generator=g, device="cuda", dtype=torch.float64)   # noqa: E731
        m = torch.arange(1, case["cap"] + 1, device="cuda", dtype=torch.float64)[None, :]
        s, w, rate, size = 0.05 + 0.45 * u(), 1.0 + 99.0 * u(), torch.exp(-7.0 * u()), torch.exp(-12.0 * u())
        R = lambda k: size * (1.0 - torch.exp(-rate * 3.0 * k / (s * k + w)))   # noqa: E731
        gain = torch.where(u() < 0.1, torch.zeros_like(R(m)), torch.clamp_min(R(m) - R(m - 1.0), 0.0))
        st["gain"] = torch.cummin(gain, 1).values.contiguous()
        st["alloc"] = torch.zeros(n, dtype=torch.int32, device="cuda")
        st["reduction"] = torch.zeros(n, dtype=torch.float64, device="cuda")
        return st

    j = _Jobs(case, seed)
    off, losses = _host(j.offsets), _host(j.losses, case["pinned"])
    k_last, past, s, w = _host(j.k_last), _host(j.m_past), _host(j.s), _host(j.w)
    ids = np.arange(n, dtype=np.int32)
    if kind == "sharded":
        st["shards"], st["exchange"] = [], slaq.LocalExchange()
        cut = [n * r // case["shards"] for r in range(case["shards"] + 1)]
        for lo, hi in zip(cut[:-1], cut[1:]):
            sh = _scheduler(case, hi - lo)
            sh.load_histories(ids[: hi - lo], off[lo: hi + 1] - off[lo], losses[off[lo]: off[hi]], k_last[lo:hi],
                              past[lo:hi], packed=case["packed"])
            sh.set_time_model(ids[: hi - lo], s[lo:hi], w[lo:hi])
            st["shards"].append(sh)
        return st

    sched = st["sched"] = _scheduler(case, n)
    st["n"] = n
    if kind == "restart":
        st.update(ids=ids, off=off, losses=losses, k_last=k_last, past=past, s=s, w=w, packed=case["packed"],
                  out=np.empty(n, np.int32))
        return st
    sched.load_histories(ids, off, losses, k_last, past, packed=case["packed"])
    if case["law"] == "fixed":
        sched.set_time_model(ids, s, w)
    if case["options"]:
        # two jobs in five come with the loss their owner expects to reach: near the curve's floor, or above it
        newest = j.losses[j.offsets[1:] - 1]
        share = torch.rand(n, generator=j.g, device="cuda", dtype=torch.float64)
        hint = torch.where(share < 0.4, newest * (0.5 + share), torch.full_like(newest, math.nan))
        sched.set_target_loss(ids, _host(hint))
    if kind in ("loop", "device"):
        # The losses still to come.  They walk along every job's curve and then start over, so that the jobs stay in
        # training however long the loop runs: of a ring, one window in four or fewer shows such a restart.
        steps = max(8, min(4 * case["hist"], 4_000_000 // n))
        every = torch.arange(n, device="cuda")
        feed = torch.stack([j.noisy(every, j.k_last + 1 + t) for t in range(steps)])
        used = [1, 2, 4, 8]
        st["steps"] = steps
        if kind == "device":
            st["d_ids"], st["d_feed"] = torch.arange(n, dtype=torch.int32, device="cuda"), list(feed)
            st["d_time"] = [_samples(j, c) for c in used]
            st["d_used"] = [torch.full((n,), c, dtype=torch.int32, device="cuda") for c in used]
            st["d_alloc"] = torch.zeros(n, dtype=torch.int32, device="cuda")
        else:
            pin = case["pinned"]
            st["ids"] = _host(torch.arange(n, dtype=torch.int32, device="cuda"), pin)
            st["feed"] = list(_host(feed, pin))
            st["time"] = [_host(_samples(j, c), pin) for c in used]
            st["used"] = [_host(torch.full((n,), c, dtype=torch.int32, device="cuda"), pin) for c in used]
            st["out"] = _host(torch.zeros(n, dtype=torch.int32, device="cuda"), pin)
            for t in range(4 if case["law"] == "samples" else 0):   # the jobs' earlier iteration times
                sched.append_losses(st["ids"], st["feed"][t - 4], st["time"][t], st["used"][t])
    elif kind == "epoch":
        st["d_alloc"] = torch.zeros(n, dtype=torch.int32, device="cuda")
    elif kind == "checkpoint":
        if case["law"] == "samples":
            for c in (1, 4):
                sched.append_losses(ids, _host(j.noisy(torch.arange(n, device="cuda"), j.k_last + 1)),
                                    _host(_samples(j, c)), np.full(n, c, np.int32))
        sched.schedule(st["T"], cores)   # the curves of an epoch are part of the state
        st["other"] = slaq.Scheduler(n, case["hist"], case["cap"])
        st["out"] = np.empty(n, np.int32)
    return st


def run(st):
    kind = st["kind"]
    if kind == "loop":
        t = st["at"]
        st["at"] = t + 1 if t + 1 < st["steps"] else 0
        st["sched"].append_losses(st["ids"], st["feed"][t], st["time"][t & 3], st["used"][t & 3])
        return st["sched"].schedule(st["T"], st["C"], out_alloc=st["out"])
    if kind == "device":
        t = st["at"]
        st["at"] = t + 1 if t + 1 < st["steps"] else 0
        st["sched"].append_losses_device(st["d_ids"], st["d_feed"][t], st["d_time"][t & 3], st["d_used"][t & 3])
        st["sched"].schedule_device(st["T"], st["C"], st["d_alloc"])
        return st["d_alloc"]
    if kind == "epoch":
        st["sched"].schedule_device(st["T"], st["C"], st["d_alloc"])
        return st["d_alloc"]
    if kind == "restart":
        st["sched"].load_histories(st["ids"], st["off"], st["losses"], st["k_last"], st["past"], packed=st["packed"])
        st["sched"].set_time_model(st["ids"], st["s"], st["w"])
        return st["sched"].schedule(st["T"], st["C"], out_alloc=st["out"])
    if kind == "predict":
        alloc, _ = st["sched"].schedule(st["T"], st["C"])
        p = st["sched"].get_predictions(want_gain=True)
        return {"alloc": alloc, "reduction": p["R"], "gain": p["gain"], "largest": p["M"], "status": p["status"]}
    if kind == "checkpoint":
        blob = st["sched"].export_state()
        st["other"].import_state(blob)
        alloc, _ = st["other"].schedule(st["T"], st["C"], out_alloc=st["out"])
        return {"bytes": int(blob.size), "alloc": alloc}
    if kind == "sharded":
        return slaq.schedule_sharded(st["shards"], st["exchange"], st["T"], st["C"])
    slaq.allocate_static(st["gain"], st["C"], st["alloc"], st["reduction"])
    return st["alloc"], st["reduction"]


def work(case):
    n, cap = case["jobs"], case["cap"]
    if case["kind"] == "allocate":
        return {"bytes": 8.0 * n * cap + 12.0 * n, "flops": 1.0 * n * cap}
    points = n * (0.8 * case["hist"] + 0.8 if case["stages"] else 0.5 * (case["hist"] + 3.0))
    # sweeps a family takes: nearly all of its trials (most fits end on the trial limit), and the starting point's
    sweeps = 1.0 + 0.9 * (5 if case["warm"] else 20)
    flops = points * (FLOP_SWEEPS * sweeps + FLOP_SETUP) + FLOP_GAIN * n * cap
    moved = 8.0 * points + 4.0 * n                       # the histories in, the allocation out
    if case["kind"] in ("loop", "device"):
        moved += 24.0 * n + 16.0 * n                     # ids, losses, times, cores; the loss and time sums stored
    elif case["kind"] == "restart":
        moved += 8.0 * points + 44.0 * n                 # the histories stored, ids, offsets, k, largest, time laws
    elif case["kind"] == "predict":
        moved += 8.0 * n * cap + 77.0 * n                # gain rows and per-job records out
    elif case["kind"] == "checkpoint":
        moved += 3 * 8.0 * points + 2 * 320.0 * n        # windows and per-job records out, in and stored
    return {"bytes": moved, "flops": flops}


def tolerance(case):
    # Predictions agree to 1e-6 between correct implementations of an unfinished fp64 iteration; cores move between
    # jobs only where gains compete within rounding.
    return {"rel": 1e-6, "max": 1e-4, "differ": 1e-3}
