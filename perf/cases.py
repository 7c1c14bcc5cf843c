"""The work that users of this package have it do, as cases that can be timed and compared.

A case is one use of the library's entry points (the methods of `binding.Hadfl`, which are the C calls):

  "watched"  a coordinator that follows every round, as `paper_2111_08274_b200.run` does: the selection
             probabilities, one fused round, its statistics and the counters read back
  "round"    one fused round, enqueued: the benchmark's step
  "rounds"   a run of consecutive rounds given to the library in one call, then its statistics
  "calls"    the same rounds as the paper's separate calls: local steps, selection, aggregation,
             the send or the mix on global-synchronisation rounds, statistics
  "backup"   rounds whose statistics and aggregated model travel to the host while the next one runs:
             the benchmark's end-to-end step

Sizes are those of `workloads.py` (vectors of ResNet-18, VGG-16 and ResNet-50 size, the sweep over
2^16 .. 2^27 parameters, 4 to 32 devices), with odd lengths among the drawn ones.
"""
import numpy as np
import torch

from paper_2111_08274_b200 import runtime, workloads

STEP_TABLE = 32          # rounds of step counts that a state holds; passes walk over them
RATIOS = (1, 1, 2, 2, 4, 4, 8, 8)   # compute-power ratios of the workloads

STORAGE = {  # name -> dtype, m_dtype, rounding
    "fp32": (0, 0, 0),
    "bf16": (1, 0, 0),
    "bf16_m16": (1, 1, 0),
    "bf16_sr": (1, 0, 1),
    "bf16_m16_sr": (1, 1, 1),
}


def _case(name, use, n, p, k, steps, rounds=1, storage="fp32", sync_every=0, beta=1.0, scale=1.0, grad_std=1e-3):
    c = {"use": use, "devices": n, "params": p, "k": k, "steps": steps, "rounds": rounds, "storage": storage,
         "sync_every": sync_every, "beta": beta, "version_scale": scale, "grad_std": grad_std}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # Smallest: the 4-device workload of 100,000 parameters, a round at a time, the caller looking at
        # each.  Launch and call latency.
        _case("watched_small", "watched", 4, 100_000, 2, "mod4", grad_std=1e-2),
        # The same workload's ten rounds in one call.
        _case("rounds_small", "rounds", 4, 100_000, 2, "mod4", rounds=10, grad_std=1e-2),
        # The benchmark's headline: ResNet-18-sized vector, 8 devices, 1 to 8 steps each.
        _case("round_resnet18", "round", 8, 11_173_962, 4, "uniform8"),
        # VGG-16-sized vector, 16 devices of power ratios 1:2:4:8, ten rounds of which the last one
        # synchronises all devices.
        _case("rounds_vgg16", "rounds", 16, 14_728_266, 4, "ratios", rounds=10, sync_every=10, scale=1.0 / 8.0),
        # ResNet-50-sized vector, 32 devices, wide aggregation.
        _case("round_resnet50", "round", 32, 23_520_842, 8, "mod4"),
        # The sweep's middle, one step per device, eight rounds in one call.
        _case("rounds_sweep_fp32", "rounds", 16, 1 << 24, 4, "ones", rounds=8),
        # The same with bf16 parameters on a smaller vector.
        _case("rounds_sweep_bf16", "rounds", 16, 1 << 22, 4, "ones", rounds=8, storage="bf16"),
        # Reduced-precision state: bf16 parameters and momentum, stochastic rounding, power ratios.
        _case("round_bf16_stochastic", "round", 16, 1 << 25, 4, "ratios", storage="bf16_m16_sr"),
        # Largest: the sweep's end, 17 GB of replicas, one step per device.
        _case("round_largest", "round", 16, 1 << 27, 4, "ones"),
        # The headline's round as the paper's separate calls.
        _case("calls_resnet18", "calls", 8, 11_173_962, 4, "uniform8"),
        # Ragged length, bf16 parameters, separate calls; the second round mixes the aggregate into the others.
        _case("calls_ragged_mix", "calls", 6, 300_007, 2, "mod4", rounds=2, storage="bf16", sync_every=2, beta=0.25,
              grad_std=1e-2),
        # End to end: statistics and the aggregated model on the host after every round.
        _case("backup_resnet18", "backup", 8, 11_173_962, 4, "uniform8", rounds=4),
    ]


MEAN_STEPS = {"ones": 1.0, "twos": 2.0, "mod4": 2.5, "uniform2": 1.5, "uniform8": 4.5, "ratios": 3.75}


def draw(rng):
    use = rng.choice(["watched", "round", "round", "rounds", "rounds", "calls", "backup"])
    n = int(round(2 ** rng.uniform(1, 5)))
    k = int(round(2 ** rng.uniform(0, 4)))
    k = max(1, min(k, n))
    steps = rng.choice(sorted(MEAN_STEPS))
    rounds = {"rounds": rng.randint(2, 16), "calls": rng.randint(1, 3), "backup": rng.randint(2, 4)}.get(use, 1)
    storage = rng.choice(["fp32", "fp32", "fp32", "bf16", "bf16", "bf16_m16", "bf16_sr", "bf16_m16_sr"])
    p = int(2 ** rng.uniform(16, 27))
    # no more replicas, and no more local steps, than the largest listed case holds and runs
    p = min(p, int(2 ** 31 / (n * rounds * MEAN_STEPS[steps])))
    if use == "backup":
        p = min(p, 1 << 25)   # the model crosses PCIe in every round
    sync_every = rng.choice([0, 0, 1, 2, 10])
    beta = rng.choice([1.0, 1.0, 0.25, 0.5])
    return _case("", use, n, p, k, steps, rounds, storage, sync_every, beta, rng.choice([1.0, 1.0 / 8.0]))


def _step_table(case, seed):
    n, rule = case["devices"], case["steps"]
    i = np.arange(n)
    if rule == "ones":
        row = np.ones(n)
    elif rule == "twos":
        row = np.full(n, 2)
    elif rule == "mod4":
        row = 1 + i % 4
    elif rule == "ratios":
        row = np.array(RATIOS)[i % len(RATIOS)]
    else:
        hi = int(rule[len("uniform"):])
        return np.random.default_rng([seed, 0x57E95]).integers(1, hi + 1, size=(STEP_TABLE, n)).astype(np.int32)
    return np.tile(row, (STEP_TABLE, 1)).astype(np.int32)


class State:
    """The arena and handle of one run, and where in the run it stands."""

    def __init__(self, case, seed):
        dtype, m_dtype, rounding = STORAGE[case["storage"]]
        self.case = case
        wl = workloads.Workload("case", case["devices"], case["params"], case["k"], 1, "fixed", (1,) * case["devices"],
                                grad_std=case["grad_std"], version_scale=case["version_scale"], dtype=dtype,
                                m_dtype=m_dtype, rounding=rounding, sync_every=case["sync_every"],
                                sync_beta=case["beta"], seed=(workloads.BASE_SEED + 1_000_003 * seed) & (2 ** 64 - 1))
        self.arena = runtime.Arena(wl)
        self.h, self.ids, self.lr, self.k = self.arena.h, self.arena.ids, wl.lr, wl.k
        self.seed = self.arena.select_seed
        self.table = _step_table(case, seed)
        rounds = case["rounds"]
        # the step counts of the next calls, as the caller's arrays
        self.chunks = [np.ascontiguousarray(self.table[(np.arange(rounds) + a * rounds) % STEP_TABLE]) for a in range(8)]
        self.round = 0
        self.calls = 0
        if case["use"] == "backup":
            self.host = [torch.empty(case["params"], dtype=torch.float32).pin_memory() for _ in range(2)]

    def steps(self):
        return self.table[self.round % STEP_TABLE]

    def syncs(self):
        return bool(self.case["sync_every"]) and (self.round + 1) % self.case["sync_every"] == 0


def prepare(case, seed):
    return State(case, seed)


def _outputs(s, selected, stats=None, **more):
    versions, counters = s.h.get_versions()
    out = {"w": s.arena.w[:, : s.case["params"]], "m": s.arena.m[:, : s.case["params"]], "selected": selected,
           "versions": versions.astype(np.int64), "counters": counters.astype(np.int64)}
    if stats is not None:
        out["norm2"], out["div2"] = stats
    out.update(more)
    return out


def run(s):
    h, use = s.h, s.case["use"]
    if use == "round":
        sel = h.round(s.ids, s.steps(), s.lr, s.round, s.k, s.seed, sync_all=s.syncs())
        s.round += 1
        return _outputs(s, sel)
    if use == "watched":
        probs = h.select_probs_after(s.ids, s.steps())
        sel = h.round(s.ids, s.steps(), s.lr, s.round, s.k, s.seed, sync_all=s.syncs())
        s.round += 1
        return _outputs(s, sel, h.stats_read(), probs=probs)
    if use == "rounds":
        steps = s.chunks[s.calls % len(s.chunks)]
        sel = h.rounds(s.round, steps, s.lr, s.k, s.seed, s.case["sync_every"])
        s.round += len(steps)
        s.calls += 1
        return _outputs(s, sel, h.stats_read())
    if use == "calls":
        chosen = []
        for _ in range(s.case["rounds"]):
            h.local_step(s.ids, s.steps(), s.lr)
            sel = h.select(s.round, s.k, s.seed)
            h.aggregate(sel)
            if s.syncs() and s.k < len(s.ids):
                others = np.setdiff1d(s.ids, sel).astype(np.int32)
                if s.case["beta"] == 1.0:
                    h.broadcast(int(sel[0]), others)
                else:
                    h.integrate(int(sel[0]), others, s.case["beta"])
            h.stats_enqueue(int(sel[0]))
            s.round += 1
            chosen.append(sel)
        return _outputs(s, np.stack(chosen), h.stats_read())
    # "backup": the previous round's model has to have arrived before the next one's copy begins
    chosen, stats = [], None
    for i in range(s.case["rounds"]):
        sel = h.round(s.ids, s.steps(), s.lr, s.round, s.k, s.seed, sync_all=s.syncs())
        stats = h.stats_read()
        if i:
            h.backup_wait()
        h.backup_begin(int(sel[0]), s.host[i % 2])
        s.round += 1
        chosen.append(sel)
    h.backup_wait()
    return _outputs(s, np.stack(chosen), stats, model=s.host[(s.case["rounds"] - 1) % 2],
                    model_before=s.host[s.case["rounds"] % 2])


def work(case):
    """Bytes: a call reads the parameters and momentum it updates once and writes them once - a run of
    rounds given in one call too.  The separate calls have their own inputs and outputs each.
    flops: per element-step 20 integer operations of the generator (ten rounds of four half products and
    four xors for four elements), 6 of the Box-Muller transform and 6 of the update; 2 per selected
    element; 5 per element for the statistics."""
    dtype, m_dtype, _ = STORAGE[case["storage"]]
    ew, em = (2 if dtype else 4), (2 if m_dtype else 4)
    n, p, k, rounds, use = case["devices"], case["params"], case["k"], case["rounds"], case["use"]
    state = n * p * 2 * (ew + em)
    flops = rounds * p * (32.0 * n * MEAN_STEPS[case["steps"]] + 2.0 * k + 5.0 * n)
    if use == "rounds":
        nbytes = state
    elif use == "calls":
        nbytes = rounds * (state + 2 * k * p * ew + n * p * ew)
        if case["sync_every"]:
            per_sync = (1 + (n - k) * (1 if case["beta"] == 1.0 else 2)) * p * ew
            nbytes += rounds / case["sync_every"] * per_sync
    elif use == "backup":
        nbytes = rounds * (state + p * (ew + 4))
    else:
        nbytes = state
    return {"bytes": float(nbytes), "flops": flops}


def tolerance(case):
    """Selections, versions and counters are exact.  Parameters, momentum and statistics: about four times
    what the kernels differ by from the same rounds with the generator's normals and the statistics'
    sums in 64 bits (the CPU checker; 100,003 parameters, 4 and 8 devices, 1 to 12 rounds).  Seen with fp32
    storage: 1.0e-7 (parameters), 2.2e-7 (momentum), 9.6e-7 (squared distances); single values 1.5e-6.  With bf16
    storage a rounding decision goes the other way in up to 2 of 10,000 values and moves the value by one
    bf16 step: 8.7e-5 and 1.3e-2."""
    return {"rel": 4e-6, "max": 6e-6} if case["storage"] == "fp32" else {"rel": 3.6e-4, "max": 5e-2}
