"""What is timed: one pass through a public entry point of the library, per case.

A case is a dict of plain values.  `prepare` builds what a caller has in hand
-- a loaded code, parameters, device buffers -- from the seed alone, `run`
makes the call and returns its whole results, `work` counts what the path
cannot do without, `exact` gives 64-bit values where results are computed
real numbers.  The codes are drawn like the library's own workloads:
quasi-cyclic bases of 3 or 4 rows, Z from 16 to 512, n from 96 to 11,520,
without 4-cycles (without 6-cycles for the (3,6) codes), and general codes
given by their check rows.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2208_05795_gb300 as tsx

# results of an enumeration: per trapping set and per candidate
SETS = ("a", "b", "orbit", "count", "thr", "flags", "key_vars", "key_off")
CANDS = ("cand_vars", "cand_thr", "cand_ts", "cand_flags", "cand_decodes", "cand_iters")


def listed():
    return [
        # The tiny code of the tests and of the first configuration, whole: a call whose launches
        # and host work count as much as its decodes.
        dict(name="enum_qc96", kind="enum", decoder="nms16", mb=3, nb=6, Z=16, g8=False, csr=False, w3=False,
             K=20, base=16, s=10, size=3, cyc=0, cands=10_000),
        # Thresholds of a handful of caller-given sets without allocation, 8-bit messages: the
        # smallest call, latency alone.
        dict(name="thresholds_n576", kind="thr", decoder="nms8", mb=3, nb=6, Z=96, K=20, base=16, s=8, cands=200),
        # The PEG (1008, 504) configuration: a general (3,6) code, K = 50, 12 bisection steps; a
        # shard of its 11.7M candidates.
        dict(name="enum_csr1008", kind="enum", decoder="nms16", mb=3, nb=6, Z=168, g8=True, csr=True, w3=False,
             K=50, base=16, s=12, size=3, cyc=0, cands=150_000),
        # The 2640-node (3,6) QC configuration with 8-cycle candidates, K = 100: a shard.
        dict(name="enum_qc2640", kind="enum", decoder="nms16", mb=3, nb=6, Z=440, g8=True, csr=False, w3=False,
             K=100, base=12, s=10, size=3, cyc=8, cands=30_000),
        # A high-rate code of the batch and serving streams, check degree 15 to 20.
        dict(name="enum_qc4608", kind="enum", decoder="nms16", mb=4, nb=18, Z=256, g8=False, csr=False, w3=True,
             K=20, base=16, s=10, size=2, cyc=0, cands=12_000),
        # The largest codes of the batch: n = 11,520, check degree up to 30.
        dict(name="enum_qc11520", kind="enum", decoder="nms16", mb=4, nb=30, Z=384, g8=False, csr=False, w3=True,
             K=20, base=16, s=10, size=2, cyc=0, cands=8_000),
        # Four codes of uneven size enumerated together in one batch run.
        dict(name="batch_uneven", kind="batch", bases="16x64 19x64 20x256 25x128", K=20, base=16, s=10,
             size=2, cands=6_000),
        # Importance-sampling FER toward a found trapping set, the serving stream's sampling job.
        dict(name="isfer_n8832", kind="isfer", mb=3, nb=23, Z=384, K=20, ebn0=4.0, mu=1.0, samples=200_000),
        # Layered simulation decoder on the caller's frames, the shape of the paper's (2560, 2048) codes.
        dict(name="lnms_n2560", kind="lnms", mb=4, nb=20, Z=128, ebn0=3.5, frames=50_000),
        # The ordered list over iterations (two stages), a shard of the 2640-node code.
        dict(name="list_qc2640", kind="list", mb=3, nb=6, Z=440, g8=True, K=100, base=12, s=10, size=3, cyc=8,
             cands=3_000),
        # Single-precision sum-product on the general (1008, 504) code.
        dict(name="spa_csr1008", kind="enum", decoder="spa", mb=3, nb=6, Z=168, g8=True, csr=True, w3=False,
             K=50, base=16, s=12, size=3, cyc=0, cands=5_000),
        # Cycles of length 4 to 10 with their EMD spectrum, the shape of the paper's Table II.
        dict(name="emd_n2560", kind="emd", mb=4, nb=20, Z=128, lmax=5),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _shape(rng, nmax=11_520):
    """A 3- or 4-row base of the batch and serving streams, n from 96 to nmax; Z >= 2 nb leaves room for girth 6."""
    while True:
        mb = rng.choice((3, 4))
        nb = rng.randint(6, 30) if mb == 3 else rng.randint(8, 30)
        Z = _logint(rng, 16, 512)
        if Z >= 2 * nb and 96 <= nb * Z <= nmax:
            return mb, nb, Z


def _some(rng, lo, E, K, s):
    """A candidate count that keeps a case below the largest listed ones."""
    top = int(1.2e11 / (E * 0.65 * K * (s + 1)))
    return _logint(rng, lo, max(lo + 1, min(top, 150_000)))


def draw(rng):
    kind = rng.choice(("enum", "enum", "enum", "enum36", "thr", "batch", "isfer", "lnms", "list", "spa", "emd"))
    if kind == "enum":  # high-rate codes
        mb, nb, Z = _shape(rng)
        K, s = rng.choice((20, 20, 50)), rng.choice((10, 12))
        return dict(kind="enum", decoder=rng.choice(("nms16", "nms16", "nms8")), mb=mb, nb=nb, Z=Z, g8=False, csr=False,
                    w3=mb == 4 and rng.random() < 0.7, K=K, base=rng.choice((12, 16)), s=s, size=2, cyc=0,
                    cands=_some(rng, 500, mb * nb * Z, K, s))
    if kind == "enum36":  # (3,6) codes, quasi-cyclic or general
        csr = rng.random() < 0.5
        Z = _logint(rng, 16, 330 if csr else 512)
        K, s = rng.choice((20, 50, 100)), rng.choice((10, 12))
        return dict(kind="enum", decoder=rng.choice(("nms16", "nms16", "nms8")), mb=3, nb=6, Z=Z, g8=Z >= 100, csr=csr,
                    w3=False, K=K, base=rng.choice((12, 16)), s=s, size=3, cyc=0, cands=_some(rng, 1000, 18 * Z, K, s))
    if kind == "thr":
        mb, nb, Z = _shape(rng, 3000)
        return dict(kind="thr", decoder=rng.choice(("nms16", "nms8")), mb=mb, nb=nb, Z=Z, K=rng.choice((20, 50)),
                    base=16, s=8, cands=_logint(rng, 1, 5000))
    if kind == "batch":
        nbs = [rng.randint(16, 30) for _ in range(rng.randint(2, 4))]
        return dict(kind="batch", bases=" ".join("%dx%d" % (nb, _logint(rng, 2 * nb, 256)) for nb in nbs), K=20, base=16,
                    s=10, size=2, cands=_logint(rng, 500, 4000))
    if kind == "isfer":
        mb, nb, Z = _shape(rng, 9500)
        top = int(4e10 / (mb * nb * Z))
        return dict(kind="isfer", mb=mb, nb=nb, Z=Z, K=20, ebn0=round(rng.uniform(3.0, 5.0), 2), mu=round(rng.uniform(0.5, 1.2), 2),
                    samples=_logint(rng, 2000, max(2001, min(200_000, top // 10))))
    if kind == "lnms":
        mb, nb, Z = _shape(rng)
        return dict(kind="lnms", mb=mb, nb=nb, Z=Z, ebn0=round(rng.uniform(2.5, 5.0), 2),
                    frames=_logint(rng, 500, max(501, min(50_000, int(4.5e8 / (mb * nb * Z))))))
    if kind == "list":
        Z = _logint(rng, 64, 440)
        K = rng.choice((20, 50, 100))
        return dict(kind="list", mb=3, nb=6, Z=Z, g8=Z >= 100, K=K, base=12, s=10, size=3, cyc=0,
                    cands=_logint(rng, 500, max(501, min(6000, int(4e9 / (18 * Z * K))))))
    if kind == "spa":
        Z = _logint(rng, 32, 330)
        return dict(kind="enum", decoder="spa", mb=3, nb=6, Z=Z, g8=False, csr=rng.random() < 0.7, w3=False, K=50, base=16,
                    s=12, size=3, cyc=0, cands=_logint(rng, 200, max(201, min(5000, int(1.4e7 / (18 * Z))))))
    mb, nb, Z = rng.choice((3, 4)), rng.randint(8, 20), _logint(rng, 40, 512)
    return dict(kind="emd", mb=mb, nb=nb, Z=Z, lmax=rng.choice((4, 5)))


# ---- codes -------------------------------------------------------------------
def _shifts(rng, mb, nb, Z, w3, g8):
    """Exponents drawn column by column, a column again while it closes a 4-cycle (a 6-cycle with g8) with the ones before it."""
    while True:
        E = np.full((mb, nb), -1, dtype=np.int32)
        for j in range(nb):
            for _ in range(400):
                col = rng.integers(0, Z, mb).astype(np.int32)
                if w3 and rng.random() < 0.5:
                    col[rng.integers(0, mb)] = -1
                E[:, j] = col
                if not _short(E, j, Z, g8):
                    break
            else:
                break
        else:
            return E


def _short(E, j, Z, g8):
    """Does column j close a cycle of length 4 (or 6) with columns before it?"""
    rows = np.flatnonzero(E[:, j] >= 0)
    for x in rows:
        for y in rows:
            if x == y:
                continue
            p = np.flatnonzero((E[x, :j] >= 0) & (E[y, :j] >= 0))
            d = (E[x, p] - E[y, p]) % Z  # what a step from row x to row y through column p shifts by
            own = (E[x, j] - E[y, j]) % Z
            if (d == own).any():
                return True
            if g8:
                for z in range(E.shape[0]):
                    if z in (x, y):
                        continue
                    a = np.flatnonzero((E[x, :j] >= 0) & (E[z, :j] >= 0))
                    b = np.flatnonzero((E[z, :j] >= 0) & (E[y, :j] >= 0))
                    da, db = (E[x, a] - E[z, a]) % Z, (E[z, b] - E[y, b]) % Z
                    hit = (da[:, None] + db[None, :]) % Z == own
                    if (hit & (a[:, None] != b[None, :])).any():
                        return True
    return False


def _code(rng, mb, nb, Z, w3=False, g8=False, csr=False):
    E = _shifts(rng, mb, nb, Z, w3, g8)
    n, m = nb * Z, mb * Z
    if not csr:
        return SimpleNamespace(kind="qc", n=n, m=m, Z=Z, shifts=E, row_ptr=None, col_idx=None)
    # a general code: the same graph under a relabelling of its nodes
    pv, pc = rng.permutation(n), rng.permutation(m)
    r = np.arange(Z)
    rows = [None] * m
    for i in range(mb):
        js = np.flatnonzero(E[i] >= 0)
        cols = pv[js[:, None] * Z + (r[None, :] + E[i, js][:, None]) % Z]
        for k in range(Z):
            rows[pc[i * Z + k]] = np.sort(cols[:, k])
    ptr = np.zeros(m + 1, dtype=np.int32)
    ptr[1:] = np.cumsum([len(x) for x in rows])
    return SimpleNamespace(kind="csr", n=n, m=m, Z=0, shifts=None, row_ptr=ptr, col_idx=np.concatenate(rows).astype(np.int32))


# ---- what the caller has in hand ----------------------------------------------
def _enum_params(case, **more):
    return dict(decoder=case.get("decoder", "nms16"), K=case["K"], base_llr=case["base"], amp_steps=case["s"],
                **({"sat": 127} if case.get("decoder") == "nms8" else {}), **more)


def _bases(case):
    """A batch's codes as (columns, Z) of their 4-row bases."""
    return [tuple(int(x) for x in b.split("x")) for b in case["bases"].split()]


def prepare(case, seed):
    rng = np.random.default_rng([seed, 7])
    kind = case["kind"]
    st = {"kind": kind}
    if kind == "batch":
        p = tsx.make_params(**_enum_params(case, max_size=case["size"], cand_end=case["cands"]))
        codes = [tsx.load_code(_code(rng, 4, nb, Z, w3=True)) for nb, Z in _bases(case)]
        st["batch"] = tsx.batch_create(codes, p)
        st["room"] = [_room(case) for _ in codes]
        return st
    desc = _code(rng, case["mb"], case["nb"], case["Z"], case.get("w3", False), case.get("g8", False), case.get("csr", False))
    code = st["code"] = tsx.load_code(desc)
    if kind in ("enum", "list"):
        more = dict(list_mode=1, kstart=-1) if kind == "list" else {}
        st["params"] = tsx.make_params(**_enum_params(case, max_size=case["size"], cycle_len=case["cyc"],
                                                      cand_end=case["cands"], **more))
        st["room"] = _room(case, kind == "list", case.get("decoder") == "spa")
    elif kind == "thr":
        N = case["cands"]
        sets = np.full((N, 4), -1, dtype=np.int32)
        for i in range(N):
            k = 1 + i % 3
            sets[i, :k] = np.sort(rng.choice(desc.n, k, replace=False))
        st["sets"] = torch.from_numpy(sets).cuda()
        st["params"] = tsx.make_params(**_enum_params(case))
        st["out"] = {k: torch.empty(N, dtype=torch.int32, device="cuda") for k in ("thr", "decodes", "iters")}
    elif kind == "isfer":
        # the trapping set of lowest threshold among the code's first candidates, as a serving job has it
        v = tsx.ts_list_view(tsx.enumerate_ts(code, K=20, base_llr=16, amp_steps=10, max_size=2, cand_end=300), keys=False)
        best = int(np.argmin(v["thr"])) if len(v["thr"]) else -1
        st["T"] = np.sort(v["key_vars"][v["key_off"][best]:v["key_off"][best + 1]]) if best >= 0 else np.zeros(1, np.int32)
        st["params"] = dict(K=case["K"], ebn0_db=case["ebn0"], mu=case["mu"], n_samples=case["samples"], job_key=1000 + seed)
    elif kind == "lnms":
        # BPSK of the all-zero word over AWGN, 4-bit channel values
        n, F = desc.n, case["frames"]
        s2 = 1.0 / (2.0 * (1.0 - desc.m / n) * 10.0 ** (case["ebn0"] / 10.0))
        g = torch.Generator(device="cuda").manual_seed(seed)
        llr = torch.empty((F, n), dtype=torch.int8, device="cuda")
        for a in range(0, F, 4096):
            y = 1.0 + math.sqrt(s2) * torch.randn((min(F, a + 4096) - a, n), generator=g, device="cuda")
            llr[a:a + 4096] = (y * (2.0 / s2)).round().clamp(-7, 7).to(torch.int8)
        st["llr"] = llr
        st["out"] = {"fail": torch.empty(F, dtype=torch.uint8, device="cuda"),
                     "iters": torch.empty(F, dtype=torch.int32, device="cuda"),
                     "x": torch.empty((F, n), dtype=torch.uint8, device="cuda")}
    elif kind == "emd":
        st["lmax"] = case["lmax"]
    return st


def _room(case, list_mode=False, floats=False):
    """The caller's result arrays.  How many sets there are, and how many nodes they have, follows from
    the code: the arrays have room for them, and what is not used holds -1."""
    N = case["cands"]
    sets, nodes = (40 * N, 1500 * N) if list_mode else (N, 24 * N + 4096)
    room = {k: np.empty(sets, np.int32) for k in SETS}
    room.update(key_vars=np.empty(nodes, np.int32), key_off=np.empty(sets + 1, np.int64))
    room.update({k: np.empty((N, 4) if k == "cand_vars" else N, np.int32) for k in CANDS})
    if floats:
        room.update(thr_f=np.empty(sets, np.float32), cand_thr_f=np.empty(N, np.float32))
    return room


def _results(v, room):
    for k, to in room.items():
        x = v[k]
        if len(x) > len(to):
            raise RuntimeError("%s: %d results, room for %d" % (k, len(x), len(to)))
        to[:len(x)] = x
        to[len(x):] = -1
    return dict(room)


def run(st):
    kind = st["kind"]
    if kind in ("enum", "list"):
        v = tsx.ts_list_view(tsx.enumerate_ts(st["code"], st["params"]), keys=False)
        out = _results(v, st["room"])
        out["stats"] = {k: x for k, x in v["stats"].items() if not k.startswith("ms_")}
        return out
    if kind == "thr":
        o = st["out"]
        tsx.decode_thresholds_noalloc(st["code"], st["sets"].data_ptr(), len(st["sets"]), o["thr"].data_ptr(), None,
                                      o["decodes"].data_ptr(), o["iters"].data_ptr(), st["params"])
        return o
    if kind == "batch":
        b = st["batch"]
        tsx.batch_run(b)
        return [_results(tsx.batch_view(b, i, keys=False), st["room"][i]) for i in range(len(b))]
    if kind == "isfer":
        r = tsx.is_fer_estimate(st["code"], st["T"], record=True, **st["params"])
        r.pop("ms")
        return r
    if kind == "lnms":
        o = st["out"]
        tsx.lnms_decode(st["code"], st["llr"].data_ptr(), len(st["llr"]), o["fail"].data_ptr(), o["iters"].data_ptr(),
                        o["x"].data_ptr())
        return o
    r = tsx.emd_spectrum(st["code"], st["lmax"])
    return {"walks": r["walks"], "count2l": r["count2l"]}


# ---- what a pass cannot do without ---------------------------------------------
def work(case):
    """Bytes: inputs read once, results written once.  Operations: 12 integer (sum-product: 84 real) per
    edge update; the edge updates follow from the data, taken here as 0.65 K iterations a decode and
    s + 1 decodes a candidate (sampling and layered decoding: 6 and 12 iterations a word)."""
    kind = case["kind"]
    if kind == "batch":
        parts = [dict(case, kind="enum", mb=4, nb=nb, Z=Z) for nb, Z in _bases(case)]
        w = [work(p) for p in parts]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    mb, nb, Z = case["mb"], case["nb"], case["Z"]
    E, n = mb * nb * Z, nb * Z
    if kind in ("enum", "list", "thr"):
        N = case["cands"]
        ops = 84 if case.get("decoder") == "spa" else 12
        eu = N * (case["s"] + 1) * 0.65 * case["K"] * E
        return {"bytes": 4 * E + 36 * N, "flops": ops * eu}
    if kind == "isfer":
        return {"bytes": 4 * E + 9 * case["samples"], "flops": case["samples"] * (12 * 6 * E + 60 * n)}
    if kind == "lnms":
        return {"bytes": 4 * E + case["frames"] * (2 * n + 5), "flops": 12 * 12 * E * case["frames"]}
    # closed walks: every walk of lmax - 1 steps but the last two, which the closing condition fixes
    nodes = nb * mb * nb * (mb * nb) ** max(0, case["lmax"] - 3)
    return {"bytes": 4 * E + 8 * 7 * 128, "flops": 8 * nodes}


# ---- 64-bit values --------------------------------------------------------------
def _normals(job, s, v):
    """The standard normal of node v in samples s: Philox4x32-10 with counter (v / 4, s, 0, 0), Box-Muller, in 64 bits."""
    M = np.uint64(0xFFFFFFFF)
    c = [np.full(len(s), v >> 2, np.uint64), s.astype(np.uint64) & M, s.astype(np.uint64) >> np.uint64(32), np.zeros(len(s), np.uint64)]
    k0, k1 = job & 0xFFFFFFFF, job >> 32
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & M, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & M]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    pr = v & 2
    ua, ub = ((2.0 * (c[pr + t] >> np.uint64(9)).astype(np.float64) + 1.0) * 2.0 ** -24 for t in (0, 1))
    r = np.sqrt(-2.0 * np.log(ua))
    return r * (np.sin(2.0 * np.pi * ub) if v & 1 else np.cos(2.0 * np.pi * ub))


def exact(case, seed):
    """The log-weights of importance sampling; everything else is a whole number, or (estimates and
    sum-product thresholds) follows from decodes that plain 64-bit code does not finish in the time."""
    if case["kind"] != "isfer":
        return None
    st = prepare(case, seed)
    p, info = st["params"], st["code"].info
    s2 = 1.0 / (2.0 * (1.0 - info["m"] / info["n"]) * 10.0 ** (case["ebn0"] / 10.0))
    s = np.arange(case["samples"], dtype=np.int64)
    lw = np.zeros(len(s))
    for v in st["T"]:
        lw += _normals(p["job_key"], s, int(v)) * math.sqrt(s2) * (p["mu"] / s2) - p["mu"] ** 2 / (2.0 * s2)
    out = {k: None for k in ("fer", "var", "sum_w", "sum_w2", "n_samples", "n_fail", "decodes", "iterations", "edge_updates", "fail")}
    return dict(out, logw=lw)
