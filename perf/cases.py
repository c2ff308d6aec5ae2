"""The work that users of this library give it, as cases to measure.

A case is one pass through the public entry points: advance a lattice, a
cube, a batch of replicas or a queue of jobs by some Monte Carlo steps and
take the results -- the lattice, the counts of Eq. (H), the volume and the
enthalpy, and the recorded series where the run records one.

Kinds:
  lattice   one square lattice, its state in the caller's device memory
  resume    a checkpointed square lattice in host memory: restored, advanced,
            observed and saved again
  batch     many replicas of uneven size in one launch
  serve     a queue of jobs through the continuous-batching server
  cube      one cubic lattice, its state in the caller's device memory

``exact`` follows the volume chain (Sec. II.B step 1) in plain numpy doubles:
while no proposal would change the gate the volume does not depend on the
bonds, so V_iso and U_LJ of every step follow from the draws alone.
"""
import math

import numpy as np
import torch

from paper_2505_05919_gb300 import Batch, _capi, params, params3
from paper_2505_05919_gb300.serve import Job, Server

SQUARE = dict(q=6, T=300.0, P=0.1, rng_words=1, init=0, layered=False, record=0)
CUBE = dict(kind="cube", q=6, T=300.0, P=0.1, init=0, eta=True, record=0)


def listed():
    return [
        # a small lattice advanced a little and read, as between the decisions of a driving
        # program (tempering, an interactive scan): latency and launches
        dict(SQUARE, name="lattice_32_short", kind="lattice", L=32, steps=20),
        # the 64 x 64 state point of 1000 steps
        dict(SQUARE, name="lattice_64", kind="lattice", L=64, steps=1000),
        # a side that no tile divides and that is no multiple of 8, the two-word draws, another q
        dict(SQUARE, name="lattice_258_ragged", kind="lattice", L=258, steps=200, q=5, rng_words=2),
        # the mid-size production run, a record every 10 steps
        dict(SQUARE, name="lattice_1024_recorded", kind="lattice", L=1024, steps=1000, record=10),
        # the headline lattice
        dict(SQUARE, name="lattice_4096", kind="lattice", L=4096, steps=200),
        # the paper's own layered schedule on the square lattice
        dict(SQUARE, name="layered_1024", kind="lattice", L=1024, steps=200, layered=True),
        # a run continued from a checkpoint in host memory and saved again
        dict(SQUARE, name="resume_2048", kind="resume", L=2048, steps=100, T=270.0),
        # 256 replicas over a (T, P) grid, sides from 32 to 512
        dict(name="batch_256", kind="batch", replicas=256, low=32, high=512, odd=False, steps=1000, uneven=False),
        # an equation-of-state scan: jobs of uneven size and length through the server
        dict(name="serve_24", kind="serve", jobs=24, low=64, high=512, sweeps_low=200, sweeps_high=4000, epoch=200),
        # the order-parameter run of the cubic lattice: every step recorded
        dict(CUBE, name="cube_32_recorded", L=32, steps=500, record=1),
        # a cube with an odd side (eta identically 1)
        dict(CUBE, name="cube_51_odd", L=51, steps=200, eta=False),
        # the paper's largest cube
        dict(CUBE, name="cube_260", L=260, steps=50),
    ]


def _log_int(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def draw(rng):
    kind = rng.choice(["lattice", "lattice", "lattice", "layered", "resume", "batch", "serve", "cube", "cube", "cube"])
    point = dict(T=round(rng.uniform(270.0, 330.0), 2), P=round(rng.uniform(0.1, 50.0), 2))
    if kind in ("lattice", "layered", "resume"):
        grain = rng.choice([2, 2, 8, 64])
        side = max(16, grain * (_log_int(rng, 16, 4096) // grain))
        steps = max(1, min(_log_int(rng, 10, 1000), int(3e9) // (side * side)))
        case = dict(SQUARE, kind="lattice", L=side, steps=steps, q=rng.choice([6, 6, 6, 3, 8]),
                    rng_words=rng.choice([1, 1, 1, 2]), init=rng.choice([0, 0, 1]), record=rng.choice([0, 0, 10, 1]))
        if kind == "layered":
            case.update(layered=True)
        if kind == "resume":
            case.update(kind="resume", record=0)
        return dict(case, **point)
    if kind == "batch":
        high = rng.choice([128, 256, 512])
        return dict(kind="batch", replicas=_log_int(rng, 2, 200), low=rng.choice([16, 32, 64]), high=high,
                    odd=rng.random() < 0.4, steps=_log_int(rng, 50, 500), uneven=rng.random() < 0.5)
    if kind == "serve":
        return dict(kind="serve", jobs=rng.randint(4, 40), low=64, high=rng.choice([256, 512, 1024]),
                    sweeps_low=100, sweeps_high=rng.choice([500, 1000]), epoch=rng.choice([50, 100, 200]))
    grain = rng.choice([1, 2, 4, 8])
    side = max(8, grain * (_log_int(rng, 8, 260) // grain))
    return dict(CUBE, L=side, steps=max(1, min(_log_int(rng, 10, 500), int(8e8) // side ** 3)),
                eta=side % 2 == 0 and rng.random() < 0.8, record=rng.choice([0, 0, 1, 10]),
                q=rng.choice([6, 6, 6, 4, 8]), init=rng.choice([0, 0, 1]), **point)


def _members(case):
    """(L, T, P, steps) of the replicas or jobs of a case: a fixed mix, the same for every seed."""
    n = case.get("replicas") or case["jobs"]
    rng = np.random.default_rng(4)
    octaves = int(math.log2(case["high"] / case["low"])) + 1
    out = []
    for r in range(n):
        side = case["low"] << int(rng.integers(octaves))
        if case.get("odd"):
            side = max(2, side - 2 * int(rng.integers(0, 8)))
        if case["kind"] == "batch":
            steps = int(rng.integers(1, 9)) * case["steps"] // 8 if case["uneven"] else case["steps"]
            out.append((side, 270.0 + 4.0 * ((r // 16) % 16), 0.1 + (r % 16) * (49.9 / 15.0), max(1, steps)))
        else:
            lo, hi = math.log(case["sweeps_low"]), math.log(case["sweeps_high"])
            out.append((side, float(rng.uniform(270.0, 330.0)), float(rng.uniform(0.1, 50.0)), int(math.exp(rng.uniform(lo, hi)))))
    return out


def _params(case, seed):
    if case["kind"] == "cube":
        return params3(case["T"], case["P"], L=case["L"], q=case["q"], init=case["init"], seed=seed, eta_moves=int(case["eta"]))
    return params(case["T"], case["P"], L=case["L"], q=case["q"], init=case["init"], seed=seed, rng_words=case["rng_words"],
                  schedule=_capi.CVF_SCHED_LAYERED if case["layered"] else _capi.CVF_SCHED_CHECKERBOARD)


class _Held:
    """What a program keeps between passes; closes its handle when it goes."""

    def __init__(self, case, seed):
        self.case, self.handle, self.cube = case, None, case["kind"] == "cube"
        self.batch = self.server = None
        stream = torch.cuda.current_stream().cuda_stream
        kind = case["kind"]
        if kind == "batch":
            self.batch = Batch([params(T, P, L=L, seed=1000 * seed + r) for r, (L, T, P, _) in enumerate(_members(case))])
            self.steps = [m[3] for m in _members(case)]
        elif kind == "serve":
            self.server = Server(epoch_steps=case["epoch"])
            self.jobs = [(T, P, L, steps, 1000 * seed + r) for r, (L, T, P, steps) in enumerate(_members(case))]
        elif self.cube:
            self.buffer = torch.empty(case["L"] ** 3, dtype=torch.int32, device="cuda")
            self.handle = _capi.cvf3_create(_params(case, seed), stream, self.buffer.data_ptr())
        else:
            p = _params(case, seed)
            self.cells = case["L"] ** 2
            self.buffer = torch.empty(2 * self.cells, dtype=torch.int16, device="cuda")
            self.handle = _capi.cvf_create(p, stream, self.buffer.data_ptr())
            if kind == "resume":
                self.volume = self.cells * p.v_iso_init
                self.saved = np.empty(self.cells, np.uint16)  # the checkpoint, and where the next one goes
                self.next = np.empty(self.cells, np.uint16)
                _capi.cvf_get_state(self.handle, self.saved.ctypes.data, self.cells)

    def __del__(self):
        if self.handle:
            (_capi.cvf3_destroy if self.cube else _capi.cvf_destroy)(self.handle)
        for held in (self.batch, self.server):
            if held is not None:
                held.close()


def prepare(case, seed):
    return _Held(case, seed)


def _results(found):
    """Observables as arrays: whole numbers, the volume part, and what the bonds add to it."""
    rows = [o.as_dict() if hasattr(o, "as_dict") else o for o in found]
    return {
        "counts": np.array([[o["sweep"], o["n_hb"], o["n_hb_raw"], o["n_coop"], o["acc_sigma"], o["acc_volume"], o["g"], o["status"]]
                            + list(o["n_state"]) for o in rows], np.int64),
        "volume": np.array([[o["V_iso"], o["U_LJ"]] for o in rows]),
        "enthalpy": np.array([[o["V"], o["H"]] for o in rows]),
    }


_RECORD = np.dtype([("whole", "<i8", 6), ("volume", "<f8", 4), ("flags", "<i4", 2), ("states", "<i8", 8)])


def _series(records):
    a = np.frombuffer(b"".join(bytes(r) for r in records), _RECORD)
    return {"counts": np.concatenate([a["whole"], a["flags"].astype(np.int64), a["states"]], axis=1),
            "volume": a["volume"][:, [0, 2]], "enthalpy": a["volume"][:, [1, 3]]}


def run(state):
    case = state.case
    if case["kind"] == "batch":
        state.batch.sweep(state.steps)
        ids = list(range(len(state.steps)))
        out = _results(state.batch.observables_many(ids))
        out["state"] = np.concatenate([state.batch.state(r).reshape(-1) for r in ids]).view(np.int16)
        return out
    if case["kind"] == "serve":
        jobs = [Job(T=T, P=P, L=L, sweeps=steps, seed=seed, keep_state=True) for T, P, L, steps, seed in state.jobs]
        for job in jobs:
            state.server.submit(job)
        while state.server.busy():
            state.server.step()
        out = _results([job.observables for job in jobs])
        out["state"] = np.concatenate([job.state.reshape(-1) for job in jobs]).view(np.int16)
        return out
    if case["kind"] == "resume":
        _capi.cvf_set_state(state.handle, state.saved.ctypes.data, state.cells, state.volume, 0)
        _capi.cvf_sweep(state.handle, case["steps"], 0)
        out = _results([_capi.cvf_observables(state.handle)])
        _capi.cvf_get_state(state.handle, state.next.ctypes.data, state.cells)
        out["state"] = state.next.view(np.int16)
        return out
    if state.cube:
        _capi.cvf3_sweep(state.handle, case["steps"], case["record"])
        out = _results([_capi.cvf3_observables(state.handle)])
        out["state"] = state.buffer
        drain = _capi.cvf3_drain_series
    else:
        _capi.cvf_sweep(state.handle, case["steps"], case["record"])
        out = _results([_capi.cvf_observables(state.handle)])
        first = (_capi.cvf_state_device_ptr(state.handle) - state.buffer.data_ptr()) // 2
        out["state"] = state.buffer[first:first + state.cells]
        drain = _capi.cvf_drain_series
    if case["record"]:
        # at most one record more than the pass has periods: it may start inside one
        records, _ = drain(state.handle, case["steps"] // case["record"] + 1)
        if records:
            out["series"] = _series(records)
    return out


def work(case):
    # bytes: the lattice read once and written once, the results written; flops: integer
    # operations -- a Philox4x32-10 block has ten rounds of two widening multiplies and four
    # XORs, an update a proposal, two counts, a threshold and a compare (about ten)
    if case["kind"] in ("batch", "serve"):
        cells = sum(L * L for L, _, _, _ in _members(case))
        updates = sum(L * L * steps for L, _, _, steps in _members(case))
        return {"bytes": 4.0 * cells + 152.0 * len(_members(case)), "flops": 100.0 * updates}
    records = case["steps"] // case["record"] if case["record"] else 0
    if case["kind"] == "cube":
        cells = case["L"] ** 3
        # one block serves four updates; the eta move of a cube of eight corners costs about 100
        return {"bytes": 8.0 * cells + 152.0 * (1 + records), "flops": cells * case["steps"] * (150.0 + 25.0 * case["eta"])}
    cells = case["L"] ** 2
    return {"bytes": 4.0 * cells + 152.0 * (1 + records), "flops": cells * case["steps"] * (40.0 + 60.0 * case["rng_words"])}


def _philox(counter, seed):
    """Philox4x32-10 (Salmon et al., SC'11) of one counter for many 64-bit seeds."""
    low = np.uint64(0xFFFFFFFF)
    x = [np.full(seed.shape, c, np.uint64) for c in counter]
    k0, k1 = seed & low, seed >> np.uint64(32)
    for _ in range(10):
        a, b = x[0] * np.uint64(0xD2511F53), x[2] * np.uint64(0xCD9E8D57)
        x = [(b >> np.uint64(32)) ^ x[1] ^ k0, b & low, (a >> np.uint64(32)) ^ x[3] ^ k1, a & low]
        k0, k1 = (k0 + np.uint64(0x9E3779B9)) & low, (k1 + np.uint64(0xBB67AE85)) & low
    return x


def _volume_chain(dim, cells, T, P, seed, steps):
    """V_iso and U_LJ after each step for lattices of `cells` cells at (T, P); None where a
    proposal would change the gate, which takes the bonds to decide."""
    reach = np.arange(-6, 7)
    grid = np.stack(np.meshgrid(*[reach] * dim, indexing="ij"), -1).reshape(-1, dim)
    d2, many = np.unique((grid ** 2).sum(1), return_counts=True)
    inside = (d2 > 0) & (d2 < 36)
    d2, many = d2[inside].astype(np.float64), many[inside].astype(np.float64)

    def energy(v):
        # r^2 = |d|^2 v on the monolayer of thickness r0, r^3 = |d|^3 v in the cube
        r6 = (d2 * v[:, None]) ** 3 if dim == 2 else d2 ** 3 * (v * v)[:, None]
        return np.where(r6 < 36.0 ** 3, many * 2.0 * (1.0 / (r6 * r6) - 1.0 / r6), 0.0).sum(1)

    N, kT = cells.astype(np.float64), T * 8.31446261815324e-3 / 5.5
    Pr = P * 1e6 * (2.9e-10 ** 3) * 6.02214076e23 / 5500.0
    v0 = 2.0 ** (1.0 / 3.0) if dim == 2 else 2.0 ** 0.5
    reached = 0.01 * (N * v0)
    V = N * v0
    u = energy(V / N)
    out_v, out_u = [], []

    def uniform(high, low):
        return ((high << np.uint64(21)) | (low >> np.uint64(11))).astype(np.float64) / 2.0 ** 53

    for s in range(steps):
        r = _philox((0xFFFFFFFF, s, 0, 3), seed)
        dV = (2.0 * uniform(r[0], r[1]) - 1.0) * reached
        new = V + dV
        v = new / N
        if np.any(v >= 2.0):
            return None
        allowed = v >= 1.0
        un = energy(np.where(allowed, v, 1.0))
        ratio = np.where(allowed, new / V, 1.0)
        with np.errstate(over="ignore"):
            bound = np.exp(-(N * (un - u) + Pr * dV) / kT + N * np.log(ratio))
        accept = allowed & (uniform(r[2], r[3]) < bound)
        V, u = np.where(accept, new, V), np.where(accept, un, u)
        out_v.append(V)
        out_u.append(N * u)
    return np.stack(out_v), np.stack(out_u)


def exact(case, seed):
    if case["kind"] in ("batch", "serve"):
        m = _members(case)
        cells = np.array([x[0] ** 2 for x in m])
        T, P = np.array([x[1] for x in m]), np.array([x[2] for x in m])
        steps = np.array([x[3] for x in m])
        seeds = np.array([1000 * seed + r for r in range(len(m))], np.uint64)
        dim, record = 2, 0
    else:
        dim = 3 if case["kind"] == "cube" else 2
        cells, T, P = np.array([case["L"] ** dim]), np.array([case["T"]]), np.array([case["P"]])
        steps, seeds, record = np.array([case["steps"]]), np.array([seed], np.uint64), case["record"]
    chain = _volume_chain(dim, cells, T, P, seeds, int(steps.max()))
    if chain is None:
        return None
    V, U = chain
    last, each = steps - 1, np.arange(len(steps))
    out = {"counts": None, "volume": np.stack([V[last, each], U[last, each]], 1), "enthalpy": None, "state": None}
    if record and int(steps[0]) >= record:
        at = np.arange(record - 1, int(steps[0]), record)
        out["series"] = {"counts": None, "volume": np.stack([V[at, 0], U[at, 0]], 1), "enthalpy": None}
    return out
