"""What a user of the estimator has it do, as a list of cases that can be timed.

A code generator that has derived a stencil or lattice-Boltzmann kernel asks which launch
configuration to emit.  It hands over its candidates (address expressions, block shape,
thread folding) and takes back every candidate's data volumes and predicted time, and the
ranking.  It does that in one call from host buffers, again and again on a resident plan
(when hardware parameters or segments are explored), through the server, or from a process
that may not allocate device memory.  The cases cover those entry points, from one candidate
to 20,000, over the layouts and address spaces the estimator accepts.
"""
import math

import numpy as np
import torch

from paper_2204_14242_gb300 import binding as B
from paper_2204_14242_gb300 import workloads as W

GIB = 1 << 30


def case(name, entry, family, n, N=(0, 0, 0), radius=0, esize=8, multidim=False, arena_gib=4, requests=0):
    c = {"entry": entry, "family": family, "n": n, "nx": N[0], "ny": N[1], "nz": N[2], "radius": radius, "esize": esize,
         "multidim": multidim, "arena_gib": arena_gib, "requests": requests}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one candidate of a small kernel, from host buffers: what a generator pays when it asks
        # about a single launch configuration (latency: launches, copies, synchronisation)
        case("call_7pt", "call", "7pt", 1, (128, 128, 128), radius=1),
        # one stencil with a hand-picked list of launch configurations
        case("call_request", "call", "request", 40),
        # the 25-point sweep (every block shape and folding of one kernel), asked once
        case("call_25pt", "call", "star", 755, (640, 512, 512), radius=4),
        # the same sweep as a resident plan that is stepped again and again
        case("step_25pt", "step", "star", 755, (640, 512, 512), radius=4),
        # a lattice-Boltzmann kernel with 42 arrays, resident
        case("step_lbm", "step", "lbm", 755, (256, 256, 256), arena_gib=12),
        # many different kernels, fp32 and fp64, on domains of any (odd) size, resident
        case("step_mixed", "step", "mixed", 4000, arena_gib=40),
        # the largest call: 20,000 different candidates from host buffers to host results
        case("call_mixed", "call", "mixed", 20000, arena_gib=80),
        # a fp32 stencil on a ragged domain counted in the multi-dimensional address space
        case("step_multidim", "step", "star", 302, (509, 383, 251), radius=2, esize=4, multidim=True),
        # array-of-structures lattice: consecutive grid points lie 15 elements apart
        case("step_aos", "step", "aos", 151, (128, 128, 128)),
        # a burst of requests through the server, each ranked by itself
        case("served_burst", "served", "request", 60, arena_gib=24, requests=24),
        # a caller that may not allocate device memory: a small sweep in the library's fixed scratch
        case("noalloc_25pt", "noalloc", "star", 76, (160, 128, 96), radius=4),
        # ranking of results that came from elsewhere (several calls, several processes)
        case("rank", "rank", "mixed", 20000),
    ]


def log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["call", "call", "step", "step", "step", "served", "noalloc"])
    if kind == "served":
        return case(None, "served", "request", log_int(rng, 16, 128), arena_gib=24, requests=rng.randint(2, 32))
    if kind == "noalloc":
        return case(None, "noalloc", "star", log_int(rng, 1, 100), [rng.randint(40, 160) for _ in range(3)],
                    radius=rng.randint(1, 4), esize=rng.choice((4, 8)))
    family = rng.choice(["star", "star", "box", "lbm", "aos", "mixed", "mixed", "request"])
    if family == "mixed":
        n = log_int(rng, 16, 5000)
        return case(None, kind, family, n, arena_gib=8 + n // 100)
    if family == "request":
        return case(None, kind, family, log_int(rng, 16, 512), arena_gib=12)
    if family in ("lbm", "aos"):
        N = [log_int(rng, 64, 320) for _ in range(3)]
        return case(None, kind, family, log_int(rng, 1, 755 if family == "lbm" else 151), N, arena_gib=24)
    N = [log_int(rng, 64, 1024) for _ in range(3)]
    return case(None, kind, family, log_int(rng, 1, 755), N, radius=rng.randint(1, 4 if family == "star" else 2),
                esize=rng.choice((4, 8)), multidim=rng.random() < 0.25, arena_gib=24)


def launch_family(rng, n):
    """n launch configurations of the 755 (151 block shapes x 5 foldings), in a random order."""
    family = [(shape, v) for shape in W.block_shapes() for v in W.FOLD_VARIANTS]
    rng.shuffle(family)
    return family[:n]


def near(rng, N):
    """A domain of about this size: its x extent moved by whole 16-element steps where it is a
    multiple of 16 itself (padded or power-of-two arrays), otherwise anywhere near."""
    sx = 16 if N[0] % 16 == 0 else 1
    return (max(8, N[0] + sx * rng.randint(-1, 1)), max(4, N[1] + rng.randint(-4, 4)), max(4, N[2] + rng.randint(-4, 4)))


def candidates(c, seed):
    """The candidates of one case (one list, or one list per request)."""
    rng = W.SplitMix64(7919 * seed + 17)
    fam, n = c["family"], c["n"]
    if fam == "mixed":
        return [W.mixed_set(n, seed=1000003 * seed + 20221)]
    if fam == "request":
        out = []
        for i in range(c["requests"] or 1):
            fields, N, flops, _ = W.random_stencil(rng)
            # the requests of a burst differ in length: from n / 2 to 3 n / 2 candidates
            k = n if not c["requests"] else max(1, n // 2 + n * (7 * i % c["requests"]) // c["requests"])
            out.append([W.Config(N=N, B=shape, fields=fields, fold_axis=v[0], fold=v[1], flops_per_lup=flops)
                        for shape, v in launch_family(rng, k)])
        return out
    N = near(rng, (c["nx"], c["ny"], c["nz"]))
    if fam == "7pt":
        fields = W.copy_fields(N, W.star_offsets(1))
        return [[W.Config(N=N, B=(32, 4, 1), fields=fields, flops_per_lup=7.0, wave_blocks_override=8)]]
    if fam == "lbm":
        fields, flops = W.lbm_fields(N), 0.0
    elif fam == "aos":
        # one array of 15 components per point, pulled and written in place
        q = len(W.D3Q15)
        acc = [W.Access(-x, -y, -z, 0, k) for k, (x, y, z) in enumerate(W.D3Q15)] + \
              [W.Access(0, 0, 0, 1, k) for k in range(q)]
        fields, flops = [W.Field(8, acc, strides=(q, q * N[0], q * N[0] * N[1]))], 0.0
    else:
        offs = W.star_offsets(c["radius"]) if fam == "star" else W.box_offsets(c["radius"])
        fields, flops = W.copy_fields(N, offs, esize=c["esize"]), float(len(offs))
    return [[W.Config(N=N, B=shape, fields=fields, fold_axis=v[0], fold=v[1], flops_per_lup=flops,
                      address_mode=int(c["multidim"])) for shape, v in launch_family(rng, n)]]


class State:
    pass


def stream():
    """The one stream this program steps its plans on."""
    if not hasattr(stream, "s"):
        stream.s = torch.cuda.Stream()
    return stream.s


class DeviceArray:
    def __init__(self, ptr, shape, typestr):
        self.__cuda_array_interface__ = {"shape": shape, "typestr": typestr, "data": (ptr, False), "version": 3}


def prepare(c, seed):
    s = State()
    s.entry = c["entry"]
    s.hw = B.hw_struct(W.a100())
    if s.entry == "rank":
        # results as several calls would return them: predicted times over a few decades, with
        # many equal ones (candidates bound by the same limiter tie)
        rng = np.random.default_rng(seed)
        s.res = np.zeros(c["n"], B.RESULT)
        s.res["t_pred"] = 10.0 ** rng.uniform(-12, -9, c["n"])
        tied = rng.random(c["n"]) < 0.3
        s.res["t_pred"][tied] = 10.0 ** rng.integers(-12, -9, c["n"])[tied]
        s.ctx = B.Context(0, c["arena_gib"] * GIB)
        return s
    s.arrays = [B.marshal(cfgs) for cfgs in candidates(c, seed)]
    if s.entry != "noalloc":
        s.ctx = B.Context(0, c["arena_gib"] * GIB)
    if s.entry == "step":
        s.plan = B.Plan(s.ctx, hw=s.hw, arrays=s.arrays[0])
        n = s.plan.n
        res, order = s.plan.device_results()
        rows = torch.as_tensor(DeviceArray(res, (n, B.RESULT.itemsize // 8), "<i8"), device="cuda")
        ni, nd = len(B.RESULT_INT), len(B.RESULT_DBL)
        s.out = {"counts": rows[:, :ni], "volumes": rows.view(torch.float64)[:, ni:ni + nd],
                 "limiter_status": rows.view(torch.int32)[:, 2 * (ni + nd):],
                 "order": torch.as_tensor(DeviceArray(order, (n,), "<i4"), device="cuda")}
    if s.entry == "served":
        s.server = B.Server(s.ctx, s.hw, mem_budget=16 * GIB)
    return s


def outputs(res, order):
    ni, nd = len(B.RESULT_INT), len(B.RESULT_DBL)
    rows = res.view(np.int64).reshape(len(res), -1)
    return {"counts": rows[:, :ni], "volumes": res.view(np.float64).reshape(len(res), -1)[:, ni:ni + nd],
            "limiter_status": res.view(np.int32).reshape(len(res), -1)[:, 2 * (ni + nd):], "order": order}


def run(s):
    if s.entry == "call":
        return outputs(*B.ws_estimate_batch(s.ctx, hw=s.hw, arrays=s.arrays[0]))
    if s.entry == "step":
        s.plan.execute(B.WS_MODE_BATCHED, stream())
        return s.out
    if s.entry == "noalloc":
        return outputs(*B.ws_estimate_batch_noalloc(0, hw=s.hw, arrays=s.arrays[0]))
    if s.entry == "rank":
        return B.ws_rank(s.ctx, s.res)
    # served: submit the burst, then collect every request in order
    ids = [s.server.submit(arrays=a) for a in s.arrays]
    got = []
    for rid in ids:
        rc = B.WS_EAGAIN
        while rc == B.WS_EAGAIN:
            rc, res, order = s.server.poll(rid, timeout_us=1000000)
        if rc != B.WS_OK:
            raise RuntimeError(f"request failed: status {rc}")
        got.append((res, order))
    return outputs(np.concatenate([r for r, _ in got]), np.concatenate([o for _, o in got]))


def work(c):
    """Descriptors in (candidates, fields, accesses), results and order out; the model's fp64
    operations.  What lies between is counting, which has no bytes it cannot do without."""
    n = c["n"] * (c["requests"] or 1)
    lists = {"7pt": (2, 8), "star": (2, 6 * c["radius"] + 2), "box": (2, (2 * c["radius"] + 1) ** 3 + 1),
             "lbm": (42, 84), "aos": (1, 30)}
    if c["entry"] == "rank":
        return {"bytes": n * (B.RESULT.itemsize + 4), "flops": 0}
    if c["family"] == "mixed":
        inputs = n * (64 + 12 * 56 + 36 * 24)      # about 11 arrays and 35 offsets per kernel, a store
    elif c["family"] == "request":
        inputs = n * 64 + max(1, c["requests"]) * (12 * 56 + 36 * 24)
    else:
        f, a = lists[c["family"]]
        inputs = n * 64 + f * 56 + a * 24
    return {"bytes": inputs + n * (B.RESULT.itemsize + 4), "flops": 60 * n}


# ---- a single candidate by enumeration: every address of every thread, sorted and made unique ----
def exact(c, seed):
    if c["entry"] == "rank" or c["n"] > 2 or c["requests"]:
        return None
    hw = W.a100()
    cfgs = candidates(c, seed)[0]
    if any(cfg.address_mode for cfg in cfgs) or len(cfgs[0].fields) > 4 or len(cfgs[0].fields[0].accesses) > 50:
        return None
    rows = [enumerate_candidate(cfg, hw) for cfg in cfgs]
    t = np.array([r["t_pred"] for r in rows])
    m, e = np.frexp(t)
    key = np.ldexp(np.rint(np.ldexp(m, 40)), e - 40)
    return {"counts": np.array([[r[k] for k in B.RESULT_INT] for r in rows], np.int64),
            "volumes": np.array([[r[k] for k in B.RESULT_DBL] for r in rows], np.float64),
            "limiter_status": np.array([[r["limiter"], 0] for r in rows], np.int32),
            "order": np.argsort(key, kind="stable").astype(np.int32)}


def enumerate_candidate(c, hw):
    fold = [1, 1, 1]
    if c.fold_axis:
        fold[c.fold_axis] = c.fold
    g = [-(-c.N[d] // (c.B[d] * fold[d])) for d in range(3)]
    T = c.B[0] * c.B[1] * c.B[2]
    nw = -(-T // 32)
    per_sm = min(hw.max_blocks_sm, hw.max_threads_sm // (32 * nw))
    total, W_ = g[0] * g[1] * g[2], c.wave_blocks_override or hw.sms * per_sm
    n = min(W_, total)
    rep = g[0] // 2 + g[0] * (g[1] // 2 + g[1] * (g[2] // 2))
    first = min(W_ * (rep // W_), total - n)
    wave = np.arange(first, first + n)
    y = np.setdiff1d(wave[(wave // g[0]) % g[1] >= 1] - g[0], wave)
    z = np.setdiff1d(np.setdiff1d(wave[wave // (g[0] * g[1]) >= 1] - g[0] * g[1], wave), y)
    r = {k: 0 for k in B.RESULT_INT}
    r.update(wave_blocks=n, wave_first_block=first, blocks_per_sm=per_sm,
             y_dist_blocks=int(first - y[0]) if len(y) else 0, z_dist_blocks=int(first - z[0]) if len(z) else 0)
    threads = {}
    for name, ids in (("rep", np.array([rep])), ("wave", wave), ("y", y), ("z", z)):
        b, t = (v.ravel() for v in np.meshgrid(ids, np.arange(nw * 32), indexing="ij"))
        p = [(b % g[0]) * c.B[0] + t % c.B[0], ((b // g[0]) % g[1] * c.B[1] + (t // c.B[0]) % c.B[1]) * fold[1],
             (b // (g[0] * g[1]) * c.B[2] + t // (c.B[0] * c.B[1])) * fold[2]]
        ok = (t < T) & (p[0] < c.N[0]) & (p[1] < c.N[1]) & (p[2] < c.N[2])
        kv = np.where(ok, np.minimum(c.fold, c.N[c.fold_axis] - p[c.fold_axis]) if c.fold_axis else 1, 0)
        threads[name] = p, kv, np.searchsorted(ids, b) * nw + t // 32, t % 32
    r["lups_block"], r["lups_wave"] = int(threads["rep"][1].sum()), int(threads["wave"][1].sum())
    unit = [0, 0, 0]
    if c.fold_axis:
        unit[c.fold_axis] = 1
    for f in c.fields:
        sets = {}
        for name, (p, kv, warp, lane) in threads.items():
            for store in ((0, 1) if name in ("rep", "wave") else (0,)):
                need = {}      # folded offset -> the folded points that need it
                for a in f.accesses:
                    if bool(a.is_store) == bool(store):
                        for k in range(c.fold):
                            o = (a.dx + k * unit[0], a.dy + k * unit[1], a.dz + k * unit[2], a.dc)
                            need[o] = min(k, need.get(o, k))
                addrs = [np.zeros(0, np.int64)]
                for o, k in need.items():
                    on = kv > k
                    adr = f.align + f.elem_bytes * (sum(f.strides[d] * (p[d] + o[d]) for d in range(3)) +
                                                    f.const_off + o[3])[on]
                    addrs.append(adr)
                    if name in ("rep", "wave") and (store or name == "rep"):
                        per_warp = len(np.unique(np.stack([warp[on], adr // 32]), axis=1).T)
                        key = "wave_store_req_sectors" if name == "wave" else \
                            "l1_store_sectors" if store else "l1_req_sectors"
                        r[key] += per_warp
                    if name == "rep":
                        half = warp[on] * 2 + lane[on] // 16
                        for h in np.unique(half):
                            words = np.unique(adr[half == h] // hw.bank_bytes)
                            while len(words):
                                group = words[(words - words[0]) * hw.bank_bytes < hw.pair_dist_bytes]
                                r["l1_bank_cycles"] += int(np.bincount(group % hw.banks).max())
                                words = words[len(group):]
                adr = np.concatenate(addrs)
                sets[name, store] = np.unique(adr // 32), np.unique(adr // 128)
        for level, pre in (("rep", "blk"), ("wave", "wave")):
            for store, kind in ((0, "load"), (1, "store")):
                r[f"{pre}_{kind}_sectors"] += len(sets[level, store][0])
                r[f"{pre}_{kind}_lines"] += len(sets[level, store][1])
        w, sy, sz = (sets[k, 0] for k in ("wave", "y", "z"))
        r["ov_y"] += len(np.intersect1d(w[0], sy[0]))
        r["ov_z"] += len(np.setdiff1d(np.intersect1d(w[0], sz[0]), sy[0]))
        r["y_lines"] += len(sy[1])
        r["z_lines"] += len(sz[1])

    def hit(i, o):
        return hw.hit[i][0] * math.exp(-hw.hit[i][1] * math.exp(-hw.hit[i][2] * o)) if hw.capacity_model else 1.0

    lb, lw = r["lups_block"], r["lups_wave"]
    r["v_l1"], v_comp = 32 * r["l1_req_sectors"] / lb, 32 * r["blk_load_sectors"] / lb
    r["o_l1"] = 128 * r["blk_load_lines"] * per_sm / hw.l1_bytes
    r["v_l2_load"] = v_comp + (1 - hit(0, r["o_l1"])) * (r["v_l1"] - v_comp)
    r["v_l2_store"] = 32 * r["l1_store_sectors"] / lb
    alloc = 128 * r["wave_load_lines"] / n
    r["o_y"], r["o_z"] = r["y_dist_blocks"] * alloc / hw.l2_bytes, r["z_dist_blocks"] * alloc / hw.l2_bytes
    r["o_st"] = 128 * r["wave_store_lines"] / hw.l2_bytes
    saved = 32 * (hit(1, r["o_y"]) * r["ov_y"] + hit(2, r["o_z"]) * r["ov_z"])
    partial = 32 * (r["wave_store_req_sectors"] - r["wave_store_sectors"])
    r["v_dram_load"] = (32 * r["wave_load_sectors"] - saved + (1 - hit(3, r["o_st"])) * partial) / lw
    r["v_dram_store"] = 32 * r["wave_store_sectors"] / lw
    r["t_l1"] = r["l1_bank_cycles"] / lb / (hw.clock_hz * hw.sms)
    r["t_l2"] = (r["v_l2_load"] + r["v_l2_store"]) / hw.bw_l2
    r["t_dram"] = (r["v_dram_load"] + r["v_dram_store"]) / hw.bw_dram
    r["t_fp"] = c.flops_per_lup / hw.fp_peak
    limits = [r["t_l1"], r["t_l2"], r["t_dram"], r["t_fp"]]
    r["t_pred"] = max(limits)
    r["limiter"] = limits.index(r["t_pred"])
    r["glups"] = 1e-9 / r["t_pred"]
    return r
