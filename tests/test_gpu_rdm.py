"""Energy functional E(h, V; c) and its density-matrix gradient on the GPU, through the C ABI, against the
oracle (which builds the density matrices by applying the operators), exact diagonalisation, a
brute-force count of connected pairs, and central finite differences (E is linear in h and V, so the
differences are exact up to rounding)."""
from __future__ import annotations

import ctypes
import functools
import os
import subprocess

import numpy as np
import pytest

import bruteforce as bf
from oracle.oracle import Oracle
from paper_1305_6981_gb300 import _native, synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _dev(x):
    return torch.as_tensor(np.ascontiguousarray(x)).to("cuda")


def _functional(system, dets, c):
    from paper_1305_6981_gb300 import EnergyFunctional
    return EnergyFunctional(system.n_elec, system.n_orb, dets, c)


def _count_pairs(dets):
    """Brute-force numbers of single- and double-excitation pairs (unordered, distinct determinants)."""
    ints = [bf.from_words(w) for w in dets]
    ns = nd = 0
    for a in range(len(ints)):
        for b in range(a + 1, len(ints)):
            x = bin(ints[a] ^ ints[b]).count("1")
            ns += x == 2
            nd += x == 4
    return ns, nd


def test_full_space_ground_state_8e8o():
    s = synth.tiny_8e8o()
    space = bf.basis(8, 4, 4)
    H = bf.hamiltonian(8, s.h, s.eri_s8, space)
    w, v = np.linalg.eigh(H)
    dets = np.array([bf.to_words(d, 1) for d in space])
    f = _functional(s, dets, v[:, 0])
    E = float(f.energy(_dev(s.h), _dev(s.eri_s8)))
    gh, ge = f.gradient(torch.ones((), dtype=torch.float64, device="cuda"))
    Eq, ghq, geq = Oracle(s, tau=0.01).rdm_energy(dets, v[:, 0])
    assert abs(E - w[0]) < 1e-10
    assert abs(E - Eq) < 1e-11
    assert np.abs(gh.cpu().numpy() - ghq).max() < 1e-12
    assert np.abs(ge.cpu().numpy() - geq).max() < 1e-12
    f.close()


@pytest.mark.parametrize("n", [600, 3000, 10000])
def test_sampled_vector_16e40o_matches_oracle(n):
    s = synth.rdm_16e40o()
    dets, c = synth.sampled_vector(s, n, seed=5)
    f = _functional(s, dets, c)
    E = float(f.energy(_dev(s.h), _dev(s.eri_s8)))
    gh, ge = f.gradient(torch.ones((), dtype=torch.float64, device="cuda"))
    Eq, ghq, geq = Oracle(s, tau=0.01).rdm_energy(dets, c)
    assert abs(E - Eq) <= 1e-12 * abs(Eq)
    assert np.abs(gh.cpu().numpy() - ghq).max() < 1e-12
    assert np.abs(ge.cpu().numpy() - geq).max() < 1e-12
    if n <= 600:
        info = f.info()
        ns, nd = _count_pairs(dets)
        assert info["single_pairs"] == ns and info["double_pairs"] == nd
    f.close()


def test_autograd_function_and_repeatability():
    from paper_1305_6981_gb300 import rdm_energy
    s = synth.rdm_16e40o()
    dets, c = synth.sampled_vector(s, 2000, seed=6)
    f = _functional(s, dets, c)
    h = _dev(s.h).requires_grad_(True)
    eri = _dev(s.eri_s8).requires_grad_(True)
    E = rdm_energy(h, eri, f)
    (2.5 * E).backward()
    gh, ge = f.gradient(torch.tensor(2.5, dtype=torch.float64, device="cuda"))
    assert torch.equal(h.grad, gh) and torch.equal(eri.grad, ge)
    E2 = f.energy(h.detach(), eri.detach())
    assert float(E2) == float(E.detach())  # fixed reduction order
    f.close()


def test_finite_differences_and_linearity_at_scale():
    """2e5 determinants of 16e/40o: E = sum h grad_h + sum V grad_eri, and central differences
    (step 1e-6) of every diagonal and 60 off-diagonal h entries and 200 ERI entries agree with the
    gradient within 1e-8."""
    s = synth.rdm_16e40o()
    dets, c = synth.sampled_vector(s, 200_000, seed=5)
    f = _functional(s, dets, c)
    h0, v0 = _dev(s.h), _dev(s.eri_s8)
    E = float(f.energy(h0, v0))
    gh, ge = f.gradient(torch.ones((), dtype=torch.float64, device="cuda"))
    lin = float((h0 * gh).sum() + (v0 * ge).sum())
    assert abs(E - lin) <= 1e-12 * abs(E)
    eps = 1e-6
    rng = np.random.default_rng(3)
    pairs = [(p, p) for p in range(40)] + [tuple(sorted(rng.choice(40, 2, replace=False))) for _ in range(60)]
    ghn = gh.cpu().numpy()
    for p, q in pairs:
        d = torch.zeros_like(h0)
        d[p, q] += eps
        if p != q:
            d[q, p] += eps
        fd = (float(f.energy(h0 + d, v0)) - float(f.energy(h0 - d, v0))) / (2 * eps)
        an = ghn[p, q] + (ghn[q, p] if p != q else 0.0)
        assert abs(fd - an) < 1e-8, (p, q, fd, an)
    gen = ge.cpu().numpy()
    for k in rng.choice(len(s.eri_s8), 200, replace=False):
        d = torch.zeros_like(v0)
        d[int(k)] = eps
        fd = (float(f.energy(h0, v0 + d)) - float(f.energy(h0, v0 - d))) / (2 * eps)
        assert abs(fd - gen[k]) < 1e-8, (k, fd, gen[k])
    f.close()


def test_full_size_million_determinants():
    """The 1e6-determinant 16e/40o vector: linearity identity and 20 sampled central differences."""
    s = synth.rdm_16e40o()
    dets, c = synth.sampled_vector(s, 1_000_000, seed=5)
    f = _functional(s, dets, c)
    h0, v0 = _dev(s.h), _dev(s.eri_s8)
    E = float(f.energy(h0, v0))
    gh, ge = f.gradient(torch.ones((), dtype=torch.float64, device="cuda"))
    assert abs(E - float((h0 * gh).sum() + (v0 * ge).sum())) <= 1e-12 * abs(E)
    assert abs(float(torch.trace(gh)) - 16.0) < 1e-10  # particle number
    eps = 1e-6
    rng = np.random.default_rng(9)
    ghn, gen = gh.cpu().numpy(), ge.cpu().numpy()
    for p, q in [(0, 0), (5, 5), (1, 2), (7, 31), (20, 39)]:
        d = torch.zeros_like(h0)
        d[p, q] += eps
        if p != q:
            d[q, p] += eps
        fd = (float(f.energy(h0 + d, v0)) - float(f.energy(h0 - d, v0))) / (2 * eps)
        assert abs(fd - (ghn[p, q] + (ghn[q, p] if p != q else 0.0))) < 1e-8
    for k in rng.choice(len(s.eri_s8), 15, replace=False):
        d = torch.zeros_like(v0)
        d[int(k)] = eps
        fd = (float(f.energy(h0, v0 + d)) - float(f.energy(h0, v0 - d))) / (2 * eps)
        assert abs(fd - gen[k]) < 1e-8
    f.close()


def _some_pairs(n_orb, n_elec, n, seed, sz=None):
    """n distinct determinants of n_elec electrons, all spins mixed (or n_alpha - n_beta = sz)."""
    rng = np.random.default_rng(seed)
    out = set()
    while len(out) < n:
        if sz is None:
            occ = rng.choice(2 * n_orb, n_elec, replace=False)
        else:
            na = (n_elec + sz) // 2
            occ = np.concatenate([2 * rng.choice(n_orb, na, replace=False), 2 * rng.choice(n_orb, n_elec - na, replace=False) + 1])
        out.add(sum(1 << int(k) for k in occ))
    return sorted(out)


def _grouping_cases():
    # two electrons share one key: whole lists in one group, below and above the records a block groups at a time,
    # and just around the size from which groups are walked as a triangle
    for n in (2, 3, 47, 48, 49, 700):
        yield f"2e-{n}", 20, 2, _some_pairs(20, 2, n, n)
    yield "2e-whole-52-orbitals", 52, 2, [(1 << a) | (1 << b) for a in range(104) for b in range(a)]
    # one key of 5,151 determinants beside keys of a hundred: an oversized partition taken in parts
    yield "3e-one-orbital-common", 52, 3, [1 | (1 << a) | (1 << b) for a in range(1, 103) for b in range(1, a)]
    # one word, all spins, the whole space; two words, many electrons, odd counts
    yield "3e-5o-whole", 5, 3, [d for d in range(1 << 10) if bin(d).count("1") == 3]
    yield "33e-40o", 40, 33, _some_pairs(40, 33, 40, 1, 1)
    yield "64e-64o-near", 64, 64, sorted({((1 << 64) - 1) ^ (1 << i) ^ (1 << (64 + a)) for i in range(0, 64, 9) for a in range(0, 64, 9)})


@pytest.mark.parametrize("case", list(_grouping_cases()), ids=lambda c: c[0])
def test_grouping_edges_match_oracle(case):
    """E and both density matrices at the sizes where the grouping changes its path, against the oracle's density
    matrices (built from operators, so lists of several S_z are right as well) and the energy they give. Every term
    is a product of two amplitudes of a unit vector and one integral: 64-bit sums of up to 1e7 terms in another order
    agree well within 1e7^(1/2) 2^-53 = 4e-13 of the largest term."""
    _, n_orb, n_elec, ints = case
    s = synth.make_system(n_orb, n_elec, seed=n_orb + n_elec, n_chol=8, fock_diagonal=False)
    W = (2 * n_orb + 63) // 64
    dets = np.array([bf.to_words(d, W) for d in ints], dtype=np.uint64)
    c = np.random.default_rng(len(ints)).normal(size=len(ints))
    c /= np.linalg.norm(c)
    f = _functional(s, dets, c)
    E = float(f.energy(_dev(s.h), _dev(s.eri_s8)))
    gh, ge = f.gradient(torch.ones((), dtype=torch.float64, device="cuda"))
    _, ghq, geq = Oracle(s, tau=0.01, ms2=n_elec % 2).rdm_energy(dets, c)
    Eq = float((s.h * ghq).sum() + (s.eri_s8 * geq).sum())
    assert abs(E - Eq) <= 1e-12 * max(1.0, abs(Eq))
    assert np.abs(gh.cpu().numpy() - ghq).max() < 1e-12 and np.abs(ge.cpu().numpy() - geq).max() < 1e-12
    info = f.info()
    if len(ints) <= 1000:  # connected or not: the counts are of pairs one and two spin orbitals apart
        assert (info["single_pairs"], info["double_pairs"]) == _count_pairs(dets)
    f.close()


def _matches_oracle(n_orb, n_elec, dets, c, want):
    """E and both density matrices of the library against the oracle's; want: (h, eri, gh, ge) of the oracle."""
    h, eri, ghq, geq = want
    from paper_1305_6981_gb300 import EnergyFunctional
    f = EnergyFunctional(n_elec, n_orb, dets, c)
    E = float(f.energy(_dev(h), _dev(eri)))
    gh, ge = f.gradient(torch.ones((), dtype=torch.float64, device="cuda"))
    Eq = float((h * ghq).sum() + (eri * geq).sum())
    assert abs(E - Eq) <= 1e-12 * max(1.0, abs(Eq))
    assert np.abs(gh.cpu().numpy() - ghq).max() < 1e-12 and np.abs(ge.cpu().numpy() - geq).max() < 1e-12
    if len(c) <= 1000:  # connected or not: the counts are of pairs one and two spin orbitals apart
        info = f.info()
        assert (info["single_pairs"], info["double_pairs"]) == _count_pairs(dets)
    f.close()


@functools.cache
def _short_hash_case(name):
    """(n_orb, n_elec, dets, c, oracle's values) of the lists that are grouped with short hashes."""
    if name in ("16e-600", "64e-2100"):  # the second: 4.2e6 keys, 2,048 partitions, the records scattered in two passes
        n_orb, n_elec, n = (40, 16, 600) if name == "16e-600" else (64, 64, 2100)
        s = synth.make_system(n_orb, n_elec, seed=5, n_chol=8, fock_diagonal=False)
        dets, c = synth.sampled_vector(s, n, seed=5)
        c = c / np.linalg.norm(c)
    else:
        _, n_orb, n_elec, ints = next(x for x in _grouping_cases() if x[0] == name)
        s = synth.make_system(n_orb, n_elec, seed=n_orb + n_elec, n_chol=8, fock_diagonal=False)
        dets = np.array([bf.to_words(d, (2 * n_orb + 63) // 64) for d in ints], dtype=np.uint64)
        c = np.random.default_rng(len(ints)).normal(size=len(ints))
        c /= np.linalg.norm(c)
    _, gh, ge = Oracle(s, tau=0.01, ms2=n_elec % 2).rdm_energy(dets, c)
    return n_orb, n_elec, dets, c, (s.h, s.eri_s8, gh, ge)


@pytest.fixture(scope="module")
def short_hash_library(tmp_path_factory):
    """bits -> the energy functional compiled with that many bits of a key's hash."""
    return functools.cache(lambda bits: _short_hash_build(bits, str(tmp_path_factory.mktemp("rdm"))))


def _short_hash_build(bits, where):
    so = os.path.join(where, f"librdm{bits}.so")
    subprocess.check_call([_native.nvcc(), _native.ARCH, *_native.NVCC_FLAGS, f"-DFQ_RDM_HASH_BITS={bits}", "-I" + _native.INCLUDE,
                           "-o", so, os.path.join(_native.CSRC, "fciqmc_rdm.cu")])
    full, L = _native.load(), ctypes.CDLL(so)
    for name in _native.SYMBOLS:
        if name.startswith("fciqmc_rdm_"):
            getattr(L, name).argtypes = getattr(full, name).argtypes
            getattr(L, name).restype = getattr(full, name).restype
    return L


@pytest.mark.parametrize("bits,name", [
    (5, "16e-600"),                  # every partition regrouped by the keys themselves
    (5, "3e-one-orbital-common"),    # a key of 5,151 determinants that shares its hash with other keys
    (5, "2e-whole-52-orbitals"),     # the same alone
    (5, "3e-5o-whole"), (5, "33e-40o"),
    (12, "64e-2100"),                # two scatter passes, partitions of several hashes taken in parts
])
def test_keys_that_share_their_hash(bits, name, short_hash_library, monkeypatch):
    """Keys that agree in every hash bit are told apart: the library compiled with 2^5 or 2^12 different hashes, so that
    in every partition many keys share one, against the oracle."""
    library = short_hash_library(bits)
    monkeypatch.setattr(_native, "load", lambda *a: library)
    _matches_oracle(*_short_hash_case(name))


@pytest.mark.parametrize("n", [48, 62, 63, 64, 65, 128, 129, 161, 2049, 2081])
def test_large_groups_in_shares(n):
    """One key of n determinants: a group is large from 63 on, and its rows are dealt to warps 32 at a time, in shares from
    128 partners on and at most 16 of them. The counts as well, up to 161."""
    s = synth.make_system(33, 2, seed=n, n_chol=8, fock_diagonal=False)
    dets = np.array([bf.to_words(d, 2) for d in _some_pairs(33, 2, n, n)], dtype=np.uint64)
    c = np.random.default_rng(n).normal(size=n)
    c /= np.linalg.norm(c)
    _, gh, ge = Oracle(s, tau=0.01).rdm_energy(dets, c)
    _matches_oracle(33, 2, dets, c, (s.h, s.eri_s8, gh, ge))


def test_one_key_is_spread_over_the_device():
    """E of the 5,356 determinants of two electrons in 52 orbitals, 1.4e7 pairs of one key, takes no longer than a few times
    that of a list of 4.7e7 pairs over many keys (it took 55 times as long when a key belonged to one block)."""
    from itertools import combinations

    def time_of(n_orb, n_elec):
        s = synth.make_system(n_orb, n_elec, seed=1, n_chol=8, fock_diagonal=False)
        dets = np.array([bf.to_words(sum(1 << k for k in occ), (2 * n_orb + 63) // 64) for occ in combinations(range(2 * n_orb), n_elec)],
                        dtype=np.uint64)
        f = _functional(s, dets, np.random.default_rng(1).normal(size=len(dets)))
        h, eri = _dev(s.h), _dev(s.eri_s8)
        f.energy(h, eri)
        best = np.inf
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            f.energy(h, eri)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        f.close()
        return best

    assert time_of(52, 2) < 5 * time_of(16, 4)


def test_pair_sums_of_equal_terms():
    """All 4,096 opposite-spin pairs of two electrons in 64 orbitals with equal amplitudes (of the alpha electron before
    the beta one: the sign changes where the beta orbital is the lower) and every integral 1: E = 4096. The 8.4e6 pairs
    share one key and their terms are equal, so plain additions err in one direction (48 times 2^-53 in all where a
    thread's are plain); a pair is followed by at most 8 + 4 + 16 of them, each within 2^-53, and the amplitudes' squares
    in c^T c and the last operations add four more."""
    M = 64
    dets = np.array([bf.to_words((1 << 2 * p) | (1 << 2 * q + 1), 2) for p in range(M) for q in range(M)], dtype=np.uint64)
    npair = M * (M + 1) // 2
    from paper_1305_6981_gb300 import EnergyFunctional
    sign = np.array([1.0 if p <= q else -1.0 for p in range(M) for q in range(M)])
    for c in (0.1, 0.3, 0.7):
        f = EnergyFunctional(2, M, dets, c * sign)
        E = float(f.energy(torch.zeros((M, M), dtype=torch.float64, device="cuda"),
                           torch.ones(npair * (npair + 1) // 2, dtype=torch.float64, device="cuda")))
        assert abs(E / 4096 - 1) <= (8 + 4 + 16 + 4) * 2.0 ** -53
        f.close()


@pytest.mark.parametrize("c", [0.1, 0.3, 1 / 3])
def test_occupation_sums_of_equal_terms(c):
    """4e5 determinants of seven electrons in 64 orbitals with equal amplitudes, the first spin orbital always occupied, and
    h = 1 on its orbital alone: E and the density matrix element are one plus the other spin's share. The c^2 are equal,
    so plain additions err in one direction (by 188 times 2^-53 where a warp's are plain); a term is followed by at most
    64 + 3 of them (a warp's determinants, the block's three copies) before it is compensated, and six operations more."""
    from paper_1305_6981_gb300 import EnergyFunctional
    M, n = 64, 400_000
    gen = torch.Generator(device="cuda").manual_seed(1)
    occ = torch.rand((n, 2 * M - 1), generator=gen, device="cuda").argsort(1)[:, :6] + 1
    bits = torch.zeros((n, 128), dtype=torch.bool, device="cuda").scatter_(1, occ, True)
    bits[:, 0] = True
    dets = torch.unique((bits.view(n, 2, 64).to(torch.int64) << torch.arange(64, device="cuda")).sum(-1), dim=0).contiguous()
    both = 1 + float((dets[:, 0] >> 1 & 1).double().mean())
    f = EnergyFunctional(7, M, dets, torch.full((len(dets),), c, dtype=torch.float64, device="cuda"))
    h = torch.zeros((M, M), dtype=torch.float64, device="cuda")
    h[0, 0] = 1
    npair = M * (M + 1) // 2
    E = float(f.energy(h, torch.zeros(npair * (npair + 1) // 2, dtype=torch.float64, device="cuda")))
    gh, _ = f.gradient(torch.ones((), dtype=torch.float64, device="cuda"))
    for x in (E, float(gh[0, 0])):
        assert abs(x / both - 1) <= (64 + 3 + 6) * 2.0 ** -53
    f.close()


def test_two_scatter_passes_match_oracle():
    """The same list above the 1,024 partitions that one scatter pass covers, with the library as it is."""
    _matches_oracle(*_short_hash_case("64e-2100"))


def _pair_counts(dets):
    """Numbers of pairs of determinants that are a single and a double excitation apart."""
    d = _dev(dets.view(np.int64))
    n_so = 64 * d.shape[1]
    occ = (d[:, :, None] >> torch.arange(64, device="cuda") & 1).reshape(len(d), n_so).half()
    ns = nd = 0
    for part in occ.split(4000):
        common = part @ occ.T  # whole numbers up to 64: exact
        apart = occ[0].sum() - common
        ns += int((apart == 1).sum())
        nd += int((apart == 2).sum())
    return ns // 2, nd // 2


@pytest.mark.parametrize("n_orb,n_elec,n", [(60, 24, 40_000), (32, 32, 9_000)])
def test_connected_pairs_above_one_scatter_pass(n_orb, n_elec, n):
    """More than 4.2e6 keys, so that the records are scattered in two passes, in two-word and one-word determinants: the
    pairs of members found through the keys are the connected pairs that the overlaps of the occupations give, each
    single N - 1 times and each double once."""
    assert n * n_elec * (n_elec - 1) // 2 > 1024 * 4096
    s = synth.make_system(n_orb, n_elec, seed=3, n_chol=8, fock_diagonal=False)
    dets, c = synth.sampled_vector(s, n, seed=8)
    f = _functional(s, dets, c)
    f.gradient(torch.ones((), dtype=torch.float64, device="cuda"))
    info = f.info()
    assert (info["single_pairs"], info["double_pairs"]) == _pair_counts(dets)
    f.close()


def test_counts_of_one_key_are_spread_over_the_device():
    """info() of the 8,128 determinants of two electrons in 64 orbitals (one key, 3.3e7 pairs): singles and doubles as the
    space gives them, and in a few milliseconds (27 when the key belonged to one block)."""
    import time
    from itertools import combinations
    M = 64
    dets = np.array([bf.to_words(1 << a | 1 << b, 2) for a, b in combinations(range(2 * M), 2)], dtype=np.uint64)
    s = synth.make_system(M, 2, seed=1, n_chol=4, fock_diagonal=False)
    f = _functional(s, dets, np.ones(len(dets)))
    f.gradient(torch.ones((), dtype=torch.float64, device="cuda"))
    times = []
    for _ in range(4):
        torch.cuda.synchronize()
        t = time.perf_counter()
        info = f.info()
        times.append(time.perf_counter() - t)
    n = len(dets)
    assert info["single_pairs"] == n * 2 * (2 * M - 2) // 2 and info["single_pairs"] + info["double_pairs"] == n * (n - 1) // 2
    assert min(times) < 5e-3
    f.close()
