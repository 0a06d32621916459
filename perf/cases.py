"""The work that users of this package have it do, as cases to measure.

A case is one of five kinds, each through the package's public entry points:

  walk    one FCIQMC run: a stored walker list is loaded, advanced by some iterations, and its rows, state and
          list are read back (a production run between two checkpoints; the list is put in determinant order,
          since the library gives it in no particular order)
  parts   a run divided among hash partitions on one GPU, advanced and read back the same way
  batch   uneven independent runs advanced together by one graph per launch, and read back
  energy  the energy functional of a new amplitude vector: pair structure, E, dE/dh and dE/dV by autograd
  list    estimators of a list that the caller holds on the device (the call that allocates nothing)

Sizes are those of the package's five workloads (synth) and of its tests and benchmark, and generic ones.
"""
from __future__ import annotations

import ctypes
import math
import random

import numpy as np
import torch

from paper_1305_6981_gb300 import Batch, EnergyFunctional, Fciqmc, Partitioned, _native, rdm_energy, synth

ROW_INTS = ("iteration", "nw_in", "nd_in", "c0_in", "nw_out", "nd_out", "attempts", "nulls", "spawn_events",
            "spawned_walkers", "death_walkers", "clone_walkers", "merged_entries", "aborted_walkers",
            "inserted_dets")
NAMED = {"8e8o": synth.tiny_8e8o, "12e24o": synth.init_12e24o, "24e60o": synth.large_24e60o,
         "16e40o": synth.rdm_16e40o}


# ---------------------------------------------------------------------------------------------- the cases
def listed():
    def walk(name, system, target, iterations, tau, thr, **kw):
        return dict(name=name, kind="walk", system=system, target=target, iterations=iterations, tau=tau, thr=thr, **kw)

    return [
        # the smallest calls: a few hundred determinants, plain FCIQMC, where launches and latency count
        walk("walk-8e8o-16e3", "8e8o", 1 << 14, 20, 0.01, -1, shift=0.5),
        # an ordinary initiator run in one-word determinants
        walk("walk-12e24o-1e6", "12e24o", 1_000_000, 30, 0.005, 3, shift=1.0),
        # two-word determinants, from a run that is still growing to the headline size
        walk("walk-24e60o-5e6", "24e60o", 5_000_000, 30, 0.001, 3),
        walk("walk-24e60o-1e8", "24e60o", 100_000_000, 30, 0.001, 3),
        # the options used in earnest: spin-coupled functions, an active space, hybrid walkers
        walk("walk-24e60o-hphf-5e6", "24e60o", 5_000_000, 30, 0.002, 3, option="hphf"),
        walk("walk-24e60o-cas-1e7", "24e60o", 10_000_000, 30, 0.001, 3, option="cas"),
        walk("walk-24e60o-hybrid-2e6", "24e60o", 2_000_000, 30, 0.001, 3, option="hybrid"),
        # a run spread over hash partitions
        dict(name="parts-24e60o-5e6", kind="parts", system="24e60o", target=5_000_000, iterations=40, tau=0.001,
             thr=3, parts=4),
        # uneven small runs (8e/16o to 16e/40o) advanced together
        dict(name="batch-16", kind="batch", runs=16, first=0, iterations=100, tau=0.005, thr=3),
        # energy functional and density matrices: a small vector, and a time-averaged one of a million determinants
        dict(name="energy-16e40o-3e3", kind="energy", system="16e40o", n=3_000),
        dict(name="energy-16e40o-1e6", kind="energy", system="16e40o", n=1_000_000),
        # estimators of a device list
        dict(name="list-24e60o-1e6", kind="list", system="24e60o", n=1_000_000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(("walk", "walk", "walk", "walk", "energy", "energy", "list", "batch", "parts"))
    if kind == "walk":
        system = rng.choice(("8e8o", "12e24o", "24e60o", "24e60o", "generic", "generic"))
        c = dict(kind="walk", system=system, iterations=rng.randint(3, 40), tau=0.005, thr=3)
        if system == "8e8o":
            c.update(tau=0.01, thr=-1, shift=0.5, target=_log(rng, 3_000, 1 << 15))
        elif system == "12e24o":
            c.update(shift=1.0, target=_log(rng, 20_000, 2_000_000))
        elif system == "24e60o":
            c.update(tau=0.001, target=_log(rng, 100_000, 60_000_000), thr=rng.randint(1, 4),
                     option=rng.choice(("plain", "plain", "hphf", "cas", "hybrid")))
            if c["option"] == "hybrid":
                c["target"] = min(c["target"], 10_000_000)
        else:
            n_orb = rng.randint(16, 44)
            c.update(n_orb=n_orb, n_elec=rng.randint(7, min(17, n_orb)), symmetry=rng.random() < 0.5,
                     target=_log(rng, 10_000, 3_000_000), shift=1.0)
        return c
    if kind == "energy":
        if rng.random() < 0.5:
            return dict(kind="energy", system="16e40o", n=_log(rng, 500, 700_000))
        n_orb = rng.randint(12, 60)
        return dict(kind="energy", system="generic", n_orb=n_orb, n_elec=rng.randint(5, min(20, n_orb)), symmetry=False,
                    n=_log(rng, 500, 300_000))
    if kind == "list":
        return dict(kind="list", system=rng.choice(("12e24o", "24e60o", "16e40o")), n=_log(rng, 300, 1_500_000))
    if kind == "batch":
        return dict(kind="batch", runs=rng.randint(3, 14), first=rng.randint(0, 40), iterations=10 * rng.randint(2, 12),
                    tau=0.005, thr=3)
    return dict(kind="parts", system=rng.choice(("12e24o", "24e60o")), target=_log(rng, 100_000, 1_500_000),
                iterations=rng.randint(10, 50), tau=0.001, thr=3, parts=rng.randint(2, 5))


# ---------------------------------------------------------------------------------------------- inputs
def _system(case):
    if case["system"] in NAMED:
        return NAMED[case["system"]]()
    # an own Hamiltonian of the given size, the same for every seed, as the named ones are
    n_orb, n_elec = case["n_orb"], case["n_elec"]
    return synth.make_system(n_orb, n_elec, seed=100 * n_orb + n_elec, n_chol=max(8, n_orb // 2),
                             symmetry=bool(case.get("symmetry")), name=f"{n_elec}e{n_orb}o")


def _options(case):
    option = case.get("option", "plain")
    if option == "hphf":
        return dict(hphf=True)
    if option == "cas":  # CAS(16e,40o) of 24e/60o: four orbitals frozen, sixteen deleted
        return dict(frozen_occupied=[(1 << 8) - 1, 0], frozen_empty=[0, ((1 << 32) - 1) << 24])
    if option == "hybrid":
        return dict(walker_fraction_bits=4, occupation_threshold=1.0)
    return {}


def _grow(run):
    """Advances a new run until its shift varies (its target population is reached) and a little further."""
    for _ in range(50):
        run.step(200)
        if run.estimates()["vary_shift"]:
            break
    run.step(100)


def _run_args(case, seed, target):
    # the more iterations a list grows for, the less of it sits on the reference, as in a long run
    part = 5000 if target >= 50_000_000 else 200
    return dict(target_walkers=target, initial_population=max(100, target // part), seed=seed,
                initial_shift=case.get("shift", 0.5 if target >= 50_000_000 else 1.0))


def _pinned(n, words):
    return (torch.empty((n, words), dtype=torch.int64, pin_memory=True).numpy().view(np.uint64),
            torch.empty(n, dtype=torch.int32, pin_memory=True).numpy(),
            torch.empty(n, dtype=torch.float64, pin_memory=True).numpy())


def _prepare_walk(case, seed):
    s = _system(case)
    t = case["target"]
    ms2 = s.n_elec % 2
    g = Fciqmc(s, case["tau"], case["thr"], ms2=ms2, main_capacity=max(1 << 14, t if t <= 10_000_000 else t // 4),
               spawn_capacity=max(1 << 14, t // 8), history_capacity=1 << 12, **_run_args(case, 1 + seed, t), **_options(case))
    _grow(g)
    n = g.estimates()["n_dets"]
    lists = _pinned(n, g.W)
    n = g.walkers_into(*lists)
    return dict(kind="walk", run=g, list=tuple(x[:n] for x in lists), state=g.state(), back=_pinned(_room(t), g.W),
                iterations=case["iterations"], room=_room(t))


def _prepare_parts(case, seed):
    t = case["target"]
    g = Partitioned(_system(case), case["tau"], case["thr"], n_partitions=case["parts"], main_capacity=max(1 << 14, t // 2),
                    spawn_capacity=max(1 << 14, t // 8), history_capacity=1 << 12, **_run_args(case, 1 + seed, t))
    _grow(g)
    return dict(kind="parts", run=g, iterations=case["iterations"], room=_room(t))


def _prepare_batch(case, seed):
    specs = synth.batch_systems(case["first"] + case["runs"], seed=3)[case["first"]:]
    runs, rooms = [], []
    for k, sp in enumerate(specs):
        s = synth.make_system(sp["n_orb"], sp["n_elec"], seed=sp["sys_seed"] % 100000, n_chol=sp["n_orb"] // 2)
        t = min(int(sp["target"]), 500_000)
        runs.append(Fciqmc(s, case["tau"], case["thr"], target_walkers=t, initial_population=max(100, t // 20),
                           initial_shift=1.0, seed=1000 * (1 + seed) + k, main_capacity=max(4 * t, 1 << 14),
                           spawn_capacity=max(1 << 12, t // 2), history_capacity=1 << 12))
        rooms.append(_room(t))
    b = Batch(runs, iterations_per_launch=10)
    for _ in range(8):
        b.step(10)
        if all(r.estimates()["vary_shift"] for r in runs):
            break
    b.step(5)
    return dict(kind="batch", batch=b, runs=runs, rooms=rooms, iterations=case["iterations"])


def _words(bits):
    """(n, 64 W) occupations -> (n, W) determinant words."""
    n = bits.shape[0]
    w = bits.view(n, -1, 64).to(torch.int64) << torch.arange(64, device=bits.device)
    return w.sum(-1)


def _order_key(dets):
    """One 64-bit key per determinant (a wrapping sum of the words times odd numbers)."""
    key = dets[:, 0] * -7046029254386353131
    return key + dets[:, 1] * -4417276706812531889 if dets.shape[1] == 2 else key


def _vector(s, n, seed, max_level):
    """The aufbau reference and distinct excitations of it that keep each spin's electrons, levels uniform on
    1..max_level, amplitudes +-exp(-level): the shape of a time-averaged wavefunction (synth.sampled_vector,
    drawn on the GPU). A space too small yields fewer determinants."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    M, na, nb = s.n_orb, (s.n_elec + 1) // 2, s.n_elec // 2
    W = (2 * M + 63) // 64
    kept = torch.zeros((1, W), dtype=torch.int64, device="cuda")
    ref = torch.zeros((1, 64 * W), dtype=torch.bool, device="cuda")
    ref[0, 0:2 * na:2] = True
    ref[0, 1:2 * nb:2] = True
    kept, level = _words(ref), torch.zeros(1, dtype=torch.int64, device="cuda")
    for _ in range(12):
        B = min(1 << 19, 2 * (n - len(level)) + 1024)
        for _ in range(-(-2 * (n - len(level)) // B)):
            L = torch.randint(1, max_level + 1, (B,), generator=gen, device="cuda")
            lo = (L - min(nb, M - nb)).clamp(min=0)
            hi = torch.minimum(L, torch.tensor(min(na, M - na), device="cuda"))
            ok = lo <= hi
            La = torch.minimum(lo + (torch.rand(B, generator=gen, device="cuda") * (hi - lo + 1)).long(), hi)
            bits = torch.zeros((B, 64 * W), dtype=torch.bool, device="cuda")
            for spin, nocc, cnt in ((0, na, La), (1, nb, L - La)):
                r_occ = torch.rand((B, nocc), generator=gen, device="cuda").argsort(1).argsort(1)
                r_vir = torch.rand((B, M - nocc), generator=gen, device="cuda").argsort(1).argsort(1)
                bits[:, spin:2 * nocc:2] = r_occ >= cnt[:, None]
                bits[:, 2 * nocc + spin:2 * M:2] = r_vir < cnt[:, None]
            kept = torch.cat([kept, _words(bits[ok])])
            level = torch.cat([level, L[ok]])
        # distinct determinants, in the order drawn
        key, order = torch.sort(_order_key(kept), stable=True)
        first = torch.ones_like(key, dtype=torch.bool)
        first[1:] = key[1:] != key[:-1]
        at = order[first].sort().values[:n]
        before = len(at)
        kept, level = kept[at], level[at]
        if before >= n:
            break
    sign = torch.randint(0, 2, (len(level),), generator=gen, device="cuda").double() * 2 - 1
    sign[0] = 1
    return kept.contiguous(), torch.exp(-level.double()) * sign, level


def _prepare_energy(case, seed):
    s = _system(case)
    dets, c, _ = _vector(s, case["n"], seed, 6)
    return dict(kind="energy", n_elec=s.n_elec, n_orb=s.n_orb, dets=dets, c=c,
                h=torch.as_tensor(s.h).cuda().requires_grad_(True), eri=torch.as_tensor(s.eri_s8).cuda().requires_grad_(True))


def _prepare_list(case, seed):
    s = _system(case)
    dets, _, level = _vector(s, case["n"], seed, 4)
    gen = torch.Generator(device="cuda").manual_seed(seed + 1)
    u = torch.rand(len(dets), generator=gen, device="cuda").clamp(min=1e-7)
    pops = (1 + torch.log(u) / math.log(2.0 / 3.0)).int() * torch.where(torch.rand(len(dets), generator=gen, device="cuda") < 0.5, -1, 1).int()
    pops[0] = max(1, case["n"] // 10)
    W = dets.shape[1]
    ref = np.zeros(2, dtype=np.uint64)
    ref[:W] = dets[0].cpu().numpy().view(np.uint64)
    return dict(kind="list", n_elec=s.n_elec, n_orb=s.n_orb, ref=ref, dets=dets, pops=pops.contiguous(),
                h=torch.as_tensor(s.h).cuda(), eri=torch.as_tensor(s.eri_s8).cuda(), lib=_native.load())


PREPARE = {"walk": _prepare_walk, "parts": _prepare_parts, "batch": _prepare_batch, "energy": _prepare_energy,
           "list": _prepare_list}


def prepare(case, seed):
    return PREPARE[case["kind"]](case, int(seed) % (1 << 20))


# ---------------------------------------------------------------------------------------------- one pass
def _rows(rows):
    return (np.array([[r[f] for f in ROW_INTS] for r in rows], dtype=np.int64),
            np.array([[r["shift"], r["num_in"]] for r in rows]))


def _room(target):
    """Entries that a list of this many walkers is given room for."""
    return min(2 * target, int(400 * target ** 0.55)) + 8192


def _ordered(dets, pops, hd, room):
    """A walker list read back, in an order that depends on its determinants alone, in arrays of `room` entries."""
    d = torch.from_numpy(dets.view(np.int64)).cuda(non_blocking=True)
    p = torch.from_numpy(pops).cuda(non_blocking=True)
    h = torch.from_numpy(hd).cuda(non_blocking=True)
    order = torch.argsort(_order_key(d))
    out = torch.zeros((room, d.shape[1]), dtype=torch.int64, device="cuda"), p.new_zeros(room), h.new_zeros(room)
    for o, x in zip(out, (d, p, h)):
        o[:len(order)] = x[order]
    return out


def _state(st):
    return [int(st["iteration"]), float(st["shift"]), int(st["vary_shift"]), int(st["shift_counter"]),
            int(st["nw_last_update"])]


def _run_walk(s):
    g, st, back = s["run"], s["state"], s["back"]
    g.set_walkers(*s["list"], iteration=st["iteration"], shift=st["shift"], vary=st["vary_shift"],
                  shift_counter=st["shift_counter"], nw_last_update=st["nw_last_update"])
    g.step(s["iterations"])
    rows = g.history(s["iterations"])
    n = g.walkers_into(*back)
    return dict(rows=_rows(rows), list=_ordered(*(x[:n] for x in back), s["room"]), state=_state(g.state()))


def _run_parts(s):
    g = s["run"]
    g.step(s["iterations"])
    rows = g.history(s["iterations"])
    return dict(rows=_rows(rows), list=_ordered(*g.walkers(), s["room"]))


def _run_batch(s):
    s["batch"].step(s["iterations"] // 10)
    ints, floats, dets, pops, hd = [], [], [], [], []
    for r, room in zip(s["runs"], s["rooms"]):
        i, f = _rows(r.history(s["iterations"]))
        d, p, h = _ordered(*r.walkers(), room)
        ints.append(i)
        floats.append(f)
        dets.append(torch.nn.functional.pad(d, (0, 2 - d.shape[1])))
        pops.append(p)
        hd.append(h)
    return dict(ints=np.stack(ints), floats=np.stack(floats), dets=torch.cat(dets), pops=torch.cat(pops), hd=torch.cat(hd))


def _run_energy(s):
    f = EnergyFunctional(s["n_elec"], s["n_orb"], s["dets"], s["c"])
    e = rdm_energy(s["h"], s["eri"], f)
    gh, ge = torch.autograd.grad(e, (s["h"], s["eri"]))
    f.close()
    return dict(e=e.detach(), gh=gh, ge=ge)


def _run_list(s):
    out = torch.empty(5, dtype=torch.float64, device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    _native.check(s["lib"].fciqmc_estimate_list_static(
        p(s["h"]), p(s["eri"]), s["n_elec"], s["n_orb"], s["ref"].ctypes.data_as(ctypes.POINTER(ctypes.c_uint64)),
        p(s["dets"]), p(s["pops"]), len(s["pops"]), 0, p(out), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
    return dict(counts=out[[0, 1, 2, 4]].long(), num=out[3])


RUN = {"walk": _run_walk, "parts": _run_parts, "batch": _run_batch, "energy": _run_energy, "list": _run_list}


def run(state):
    return RUN[state["kind"]](state)


# ---------------------------------------------------------------------------------------------- work and tolerance
def work(case):
    """What a pass cannot do without. Lists, once in and once out of the library; per iteration each determinant's
    words, population, diagonal element and new population once. A spawning attempt draws one Philox4x32-10 block
    (about 60 operations) and decides on one matrix element (about 60 more). Energy: the determinants, amplitudes
    and integrals read and the gradients written; per candidate pair of determinants a product and two sums, once
    for E and once for the density matrices, and 120 operations for the keys and the diagonal of a determinant."""
    kind = case["kind"]
    if kind == "energy":
        s_orb = {"16e40o": 40}.get(case["system"], case.get("n_orb"))
        ne = {"16e40o": 16}.get(case["system"], case.get("n_elec"))
        n, npair = case["n"], s_orb * (s_orb + 1) // 2
        W = (2 * s_orb + 63) // 64
        # candidate pairs grow somewhat faster than the list: 2.8e8 for a million determinants of 16e/40o
        pairs = 280.0 * n * min(1.0, (n / 1e6) ** 0.28)
        return dict(bytes=n * (8 * W + 8) + 4 * 8 * (s_orb * s_orb + npair * (npair + 1) // 2),
                    flops=10 * pairs + n * ne * (ne - 1) / 2 * 10)
    if kind == "list":
        W = 1 if case["system"] == "12e24o" else 2
        return dict(bytes=case["n"] * (8 * W + 4), flops=case["n"] * 20)
    if kind == "batch":
        specs = synth.batch_systems(case["first"] + case["runs"], seed=3)[case["first"]:]
        w = float(sum(min(int(sp["target"]), 500_000) for sp in specs))
        return dict(bytes=case["iterations"] * w * 0.05 * 28, flops=case["iterations"] * w * 120)
    # the determinants of a settled list: about one for every twenty walkers at large sizes
    w, W = float(case["target"]), 2 if case["system"] == "24e60o" or case.get("n_orb", 0) > 32 else 1
    nd = 0.05 * w
    return dict(bytes=nd * (case["iterations"] * (8 * W + 12) + 2 * (8 * W + 12)), flops=case["iterations"] * w * 120)


def tolerance(case):
    # walker lists, counters and shifts are the same to the bit whatever the order of the work (every draw is keyed
    # by determinant, attempt and iteration); the projected-energy numerators are 64-bit sums in slot order
    if case["kind"] == "energy":
        return {"rel": 1e-12, "max": 1e-11}
    return {"rel": 1e-12, "max": 1e-11}


# ---------------------------------------------------------------------------------------------- the same in plain torch
def _bits(dets, n_so):
    sh = torch.arange(64, device=dets.device)
    return ((dets[:, :, None] >> sh) & 1).reshape(len(dets), -1)[:, :n_so].bool()


def _pair_index(p, q):
    hi, lo = torch.maximum(p, q), torch.minimum(p, q)
    return hi * (hi + 1) // 2 + lo


def _eri_index(p, q, r, s):
    return _pair_index(_pair_index(p, q), _pair_index(r, s))


def _between(cum, row, k, l):
    """Occupied spin orbitals strictly between k and l (cum[., x]: occupied below x)."""
    lo, hi = torch.minimum(k, l), torch.maximum(k, l)
    return cum[row, hi] - cum[row, lo + 1].minimum(cum[row, hi])


def _two(mask):
    """Columns of the first and of the last set entry of each row."""
    m = mask.to(torch.int8)
    return m.argmax(1), mask.shape[1] - 1 - m.flip(1).argmax(1)


def _exact_energy(case, seed):
    s = _prepare_energy(case, int(seed) % (1 << 20))
    dets, c, M = s["dets"], s["c"].double(), s["n_orb"]
    N, n, n_so = s["n_elec"], len(s["c"]), 2 * s["n_orb"]
    occ = _bits(dets, n_so)
    cum = torch.nn.functional.pad(occ.to(torch.int64).cumsum(1), (1, 0))
    gh = torch.zeros(M * M, dtype=torch.float64, device="cuda")
    ge = torch.zeros(s["eri"].numel(), dtype=torch.float64, device="cuda")

    def add(to, at, x):
        to.index_add_(0, at, x)

    # diagonal: occupation pairs weighted with the squared amplitudes
    o = occ.double()
    w = o.T @ (o * (c * c)[:, None])
    p, q = torch.triu_indices(n_so, n_so, 1, device="cuda")
    P, Q = p // 2, q // 2
    k = torch.arange(n_so, device="cuda")
    add(gh, (k // 2) * (M + 1), w[k, k])
    add(ge, _eri_index(P, P, Q, Q), w[p, q])
    same = (p % 2) == (q % 2)
    add(ge, _eri_index(P, Q, Q, P)[same], -w[p, q][same])
    oh = occ.half()
    rows = max(1, min(n, (1 << 29) // n))
    for r0 in range(0, n, rows):
        left = N - (oh[r0:r0 + rows] @ oh[r0:].T)  # exact: small whole numbers
        at = ((left == 1) | (left == 2)).nonzero()
        for part in at.split(1 << 22):
            I, J = part[:, 0] + r0, part[:, 1] + r0
            keep = I < J
            I, J = I[keep], J[keep]
            holes, parts = occ[I] & ~occ[J], occ[J] & ~occ[I]
            cc = c[I] * c[J]
            i, j = _two(holes)
            a, b = _two(parts)
            one = i == j
            # singles i -> a
            i1, a1, I1 = i[one], a[one], I[one]
            sg = cc[one] * (1 - 2 * (_between(cum, I1, i1, a1) % 2)).double()
            x, y = i1 // 2, a1 // 2
            add(gh, x * M + y, sg)
            add(gh, y * M + x, sg)
            r, jj = occ[I1].nonzero(as_tuple=True)
            rest = jj != i1[r]
            r, jj = r[rest], jj[rest]
            add(ge, _eri_index(x[r], y[r], jj // 2, jj // 2), 2 * sg[r])
            ex = (jj % 2) == (i1[r] % 2)
            r, jj = r[ex], jj[ex]
            add(ge, _eri_index(x[r], jj // 2, jj // 2, y[r]), -2 * sg[r])
            # doubles i < j -> a < b
            two = ~one
            i, j, a, b, I = i[two], j[two], a[two], b[two], I[two]
            inside = lambda v: ((v > torch.minimum(j, b)) & (v < torch.maximum(j, b))).long()  # noqa: E731
            par = _between(cum, I, i, a) + _between(cum, I, j, b) - inside(i) + inside(a)
            sg = cc[two] * (1 - 2 * (par % 2)).double()
            d = ((i % 2) == (a % 2)) & ((j % 2) == (b % 2))
            e = ((i % 2) == (b % 2)) & ((j % 2) == (a % 2))
            i, j, a, b = i // 2, j // 2, a // 2, b // 2
            add(ge, _eri_index(i, a, j, b)[d], 2 * sg[d])
            add(ge, _eri_index(i, b, j, a)[e], -2 * sg[e])
    norm = (c * c).sum()
    gh, ge = (gh / norm).view(M, M), ge / norm
    return dict(e=(s["h"].detach() * gh).sum() + (s["eri"].detach() * ge).sum(), gh=gh, ge=ge)


def _exact_list(case, seed):
    s = _prepare_list(case, int(seed) % (1 << 20))
    dets, pops, M = s["dets"], s["pops"].double(), s["n_orb"]
    h, eri = s["h"], s["eri"]
    occ = _bits(dets, 2 * M)
    ref = occ[0]
    cum = torch.nn.functional.pad(ref.to(torch.int64).cumsum(0), (1, 0))[None]
    num = torch.zeros((), dtype=torch.float64, device="cuda")
    level = (ref & ~occ).sum(1)
    near = ((level == 1) | (level == 2)).nonzero()[:, 0]
    i, j = _two(ref & ~occ[near])
    a, b = _two(occ[near] & ~ref)
    z = torch.zeros_like(i)
    x = pops[near]
    one = i == j
    sign = (1 - 2 * (_between(cum, z, i, a) % 2)).double()[one]
    i1, a1 = i[one], a[one]
    v = h[i1 // 2, a1 // 2].clone()
    for k in ref.nonzero()[:, 0].tolist():
        kk = torch.full_like(i1, k)
        use = (i1 != k).double()
        v += use * eri[_eri_index(i1 // 2, a1 // 2, kk // 2, kk // 2)]
        v -= use * (i1 % 2 == k % 2).double() * eri[_eri_index(i1 // 2, kk // 2, kk // 2, a1 // 2)]
    num += (sign * v * x[one]).sum()
    i, j, a, b, x, z = i[~one], j[~one], a[~one], b[~one], x[~one], z[~one]
    inside = lambda y: ((y > torch.minimum(j, b)) & (y < torch.maximum(j, b))).long()  # noqa: E731
    sign = (1 - 2 * ((_between(cum, z, i, a) + _between(cum, z, j, b) - inside(i) + inside(a)) % 2)).double()
    d = (((i % 2) == (a % 2)) & ((j % 2) == (b % 2))).double()
    e = (((i % 2) == (b % 2)) & ((j % 2) == (a % 2))).double()
    i, j, a, b = i // 2, j // 2, a // 2, b // 2
    num += (sign * x * (d * eri[_eri_index(i, a, j, b)] - e * eri[_eri_index(i, b, j, a)])).sum()
    counts = torch.stack([pops.abs().sum().long(), torch.tensor(len(pops), device="cuda"), s["pops"][0].long(),
                          torch.tensor(0, device="cuda")])
    return dict(counts=counts, num=num)


def exact(case, seed):
    """Energies, density matrices and numerators from their definitions (dense overlaps of the occupations). The
    walker dynamics is integer and has no such value."""
    if case["kind"] == "energy" and case["n"] <= 1_000_000:
        return _exact_energy(case, seed)
    if case["kind"] == "list":
        return _exact_list(case, seed)
    return None
