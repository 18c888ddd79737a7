"""The work that a user of the library has it do, as cases that can be timed.

A case is one call of a public entry point: ``Correlators.run`` for a few time
slices of one lattice (the octet's 52 channels, coupled-channel subsets and the
decuplet, in each precision used in earnest), ``run_streamed`` from pinned host
memory, ``LatticeBatch.run`` for an uneven batch, and ``Correlators.project``
on finished correlators.  ``exact`` evaluates the same correlators from their
definition in 64 bits: sink tensors by einsum, the Wick determinant and the
source tensors as one sparse matrix per source and spin pair, the sum over X
by torch.fft.
"""
import functools
import itertools
import math

import numpy as np
import torch

from paper_1510_00903_gb300 import bbc

M_UD, M_S = 0.3, 0.4
PRECISION = {"fp64": bbc.BBC_FP64, "df64": bbc.BBC_DF64, "mixed": bbc.BBC_MIXED_FP32}
DTYPE = {"c128": torch.complex128, "c64": torch.complex64}
CHANNELS = {"octet": "0-51", "NN": "0", "LambdaN": "1-9", "S-2": "10-41", "decuplet": "64-153"}


def _ids(text):
    """Channel ids of a list by name, or of "a-b,c"."""
    out = []
    for part in CHANNELS.get(text, text).split(","):
        a, _, b = part.partition("-")
        out += range(int(a), int(b or a) + 1)
    return out


def _case(name, precision, L, T, **kw):
    case = dict(name=name, kind="run", precision=precision, L=L, T=T, t0=0, channels="octet", first=1, slices=1,
                slots=1, dtype="c128", field="gauss", lower=False, normalised=True, tuned=False)
    case.update(kw)
    return case


def listed():
    return [
        # one nucleon-nucleon channel on a toy lattice: the latency of a call
        _case("nn_L4_fp64", "fp64", 4, 8, channels="NN"),
        # coupled Lambda N - Sigma N channels: five slices through two slots (a ragged last wave), source at t0 = 5
        _case("lambda_n_L8_fp64", "fp64", 8, 15, t0=5, channels="LambdaN", first=3, slices=5, slots=2, field="smooth"),
        # the paper's 16^3 x 32 lattice, every channel, in the default precision
        _case("octet_L16_fp64", "fp64", 16, 32, slices=2, slots=2),
        # the same in the fast FP64-accurate arithmetic, launch shapes tuned as a long run does
        _case("octet_L16_df64", "df64", 16, 32, first=7, slices=4, slots=2, tuned=True),
        # S = -2 coupled channels on a lattice with a factor 3: smooth fields, complex64 files, backward propagation
        _case("s2_L24_df64", "df64", 24, 48, t0=12, channels="S-2", first=20, dtype="c64", field="smooth", lower=True),
        # production volume: one slice of 48^3 x 96, every channel
        _case("octet_L48_df64", "df64", 48, 96, first=5, dtype="c64", tuned=True),
        # throughput on the paper's lattice in single precision
        _case("octet_L16_mixed", "mixed", 16, 32, first=4, slices=8, slots=4, tuned=True),
        # a power-of-two production volume, slice by slice, raw correlators
        _case("octet_L32_mixed", "mixed", 32, 64, first=30, slices=2, dtype="c64", normalised=False, field="smooth"),
        # propagators too large to keep on the card: streamed from pinned host memory
        _case("stream_L48_mixed", "mixed", 48, 3, kind="stream", first=0, slices=3, dtype="c64"),
        # several lattices and wall sources queued as one batch
        _case("batch_mixed", "mixed", 24, 4, kind="batch", lattices="8x5,16x6,24x3", sources=2, dtype="c64"),
        # Omega Omega and p Omega (decuplet operators), all vector components
        _case("decuplet_L16_mixed", "mixed", 16, 32, channels="decuplet", first=9, slices=2, slots=2),
        # spin states and the S / D wave split of finished correlators
        _case("project_L24", "fp64", 24, 48, kind="project", slices=2),
    ]


def draw(rng):
    kind = rng.choice(["run"] * 7 + ["stream", "batch", "project"])
    precision = rng.choice(["fp64", "df64", "mixed"])
    # lattice extents spread over the supported ones; FP64 (4 times the cost of df64) stops at 24, host streaming
    # starts where it is used
    L = rng.choice([4, 8, 16, 24] if precision == "fp64" else [4, 8, 16, 24, 32, 48])
    if kind == "stream":
        L, precision = rng.choice([16, 24, 32]), rng.choice(["df64", "mixed"])
    T = rng.randint(max(3, L), 2 * L + 1)
    most = {4: 12, 8: 9, 16: 6, 24: 3, 32: 2, 48: 1}[L] if precision != "fp64" else {4: 12, 8: 7, 16: 3, 24: 1}[L]
    slices = rng.randint(1, min(most, T))
    lists = ["octet", "NN", "LambdaN", "S-2", ",".join(map(str, sorted(rng.sample(range(52), rng.randint(2, 20)))))]
    if L <= 16:
        lists.append(",".join(map(str, sorted(rng.sample(range(64, 154), rng.randint(3, 30))))))
    case = _case("", precision, L, T, kind=kind, t0=rng.randrange(T), channels=rng.choice(lists), first=rng.randrange(T),
                 slices=slices, slots=rng.randint(1, min(slices, 4)), dtype=rng.choice(["c128", "c64"]),
                 field=rng.choice(["gauss", "smooth"]), lower=rng.random() < 0.25, normalised=rng.random() < 0.75,
                 tuned=rng.random() < 0.25)
    del case["name"]
    if kind == "project":
        case.update(L=rng.choice([4, 8, 16, 24, 32]), precision="fp64", channels="octet", slices=rng.randint(1, 2))
    elif kind == "stream":
        case.update(T=slices + 1, t0=0, first=rng.randint(0, 1), slots=1)
    elif kind == "batch":
        case.update(precision="mixed", L=24, T=4, sources=rng.randint(1, 3), tuned=False, lattices=",".join(
            f"{n}x{rng.randint(2, 5)}" for n in rng.sample([4, 8, 16, 24], rng.randint(1, 3))))
    return case


# ---------------------------------------------------------------- inputs
def _times(case):
    return [(case["first"] + i) % case["T"] for i in range(case["slices"])]


def _field(gen, L, n, field, dtype):
    """n slices [n, V, 12, 12]: complex Gaussians (E|z|^2 = 1), or a Coulomb-gauge wall source's shape in outline:
    a part that barely varies over the slice, lower Dirac components a tenth of the upper ones, and noise."""
    z = torch.randn((n, L ** 3, 12, 12), generator=gen, dtype=torch.complex128, device="cuda")
    if field == "smooth":
        spin = torch.tensor([1.0] * 6 + [0.1] * 6, dtype=torch.float64, device="cuda")
        mean = torch.eye(12, dtype=torch.complex128, device="cuda") + 0.1 * torch.randn(
            (n, 1, 12, 12), generator=gen, dtype=torch.complex128, device="cuda")
        z = (mean + 0.3 * z) * (spin[:, None] * spin[None, :])
    return z.to(dtype)


def _propagators(seed, L, T, t0, times, field, dtype, lower=False):
    """Light and strange propagators of the slices `times`, each decayed by exp(-m d)."""
    gen = torch.Generator(device="cuda").manual_seed(1000003 * seed + 8191 * L + 31 * T + t0)
    out = []
    for m in (M_UD, M_S):
        S = _field(gen, L, len(times), field, torch.complex128)
        for i, t in enumerate(times):
            S[i] *= math.exp(-m * _distance(t, t0, T, lower))
        out.append(S.to(dtype))
    return out


def _distance(t, t0, T, lower):
    return (t0 - t) % T if lower else (t - t0) % T


def _lattices(case):
    return [tuple(int(x) for x in p.split("x")) for p in case["lattices"].split(",")]


def prepare(case, seed):
    dtype, kind = DTYPE[case["dtype"]], case["kind"]
    if kind == "batch":
        lat = _lattices(case)
        inputs = [tuple(_propagators(seed, L, T, 0, range(T), case["field"], dtype)) for L, T in lat]
        batch = bbc.LatticeBatch(lat, inputs, n_sources=case["sources"], channels=_ids(case["channels"]),
                                 precision=PRECISION[case["precision"]], m_ud=M_UD, m_s=M_S)
        return {"case": case, "batch": batch}
    cor = bbc.Correlators(case["L"], case["T"], case["t0"], M_UD, M_S, channels=_ids(case["channels"]),
                          precision=PRECISION[case["precision"]], slices=case["slots"],
                          components=bbc.BBC_LOWER if case["lower"] else bbc.BBC_UPPER)
    state = {"case": case, "cor": cor, "times": _times(case)}
    if kind == "project":
        state["C"] = _correlators(case, seed)
        return state
    times = list(range(case["T"])) if kind == "stream" else state["times"]
    Sl, Ss = _propagators(seed, case["L"], case["T"], case["t0"], times, case["field"], dtype, case["lower"])
    if case["tuned"]:
        cor.autotune(Sl[0], Ss[0], t=times[0], reps=2)
    if kind == "stream":
        Sl, Ss = (torch.empty(S.shape, dtype=S.dtype, pin_memory=True).copy_(S) for S in (Sl, Ss))
        # every slice's correlators, as the consumer queued after each slice keeps them
        state["kept"] = torch.empty((case["slices"], len(cor.channels), cor.V, 16), dtype=torch.complex128, device="cuda")
        state["out"] = torch.empty_like(state["kept"][0])
    state["S"] = (Sl, Ss)
    return state


def _correlators(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn((case["slices"], len(_ids(case["channels"])), case["L"] ** 3, 16), generator=gen,
                       dtype=torch.complex128, device="cuda")


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        state["batch"].run()
        return state["batch"].outputs
    cor = state["cor"]
    if case["kind"] == "project":
        return cor.project(state["C"])
    Sl, Ss = state["S"]
    if case["kind"] == "stream":
        kept = iter(state["kept"])
        cor.run_streamed(Sl, Ss, state["times"], state["out"], case["normalised"],
                         on_slice=lambda t, out: next(kept).copy_(out, non_blocking=True))
        return state["kept"]
    return cor.run(Sl, Ss, state["times"], normalised=case["normalised"])


# ---------------------------------------------------------------- work
@functools.lru_cache(maxsize=None)
def _plan_sizes(channels):
    ctx = bbc.bbc_create(2, 2, 0, M_UD, M_S, bbc.BBC_FP64, list(channels))
    try:
        return bbc.bbc_plan_sizes(ctx)
    finally:
        bbc.bbc_destroy(ctx)


def work(case):
    """Bytes: the propagators (or correlators) read once, the correlators written once.  Flops: the effective block
    algorithm's block-pair products (8 per complex multiply-add), the block rows (about 12 complex multiply-adds each
    with their tensor entries) and the Fourier transforms of blocks and correlators (5 log2 V per value)."""
    ids = _ids(case["channels"])
    if case["kind"] == "project":
        n = case["slices"] * len(ids) * case["L"] ** 3 * 16
        return {"bytes": 3 * 16 * n, "flops": 8 * n}
    size = _plan_sizes(tuple(ids))
    lattices = [(case["L"], case["slices"])]
    if case["kind"] == "batch":
        lattices = [(L, T * case["sources"]) for L, T in _lattices(case)]
    b = f = 0
    for L, n in lattices:
        V = L ** 3
        b += n * V * (2 * 144 * (16 if case["dtype"] == "c128" else 8) + len(ids) * 16 * 16)
        f += n * V * (8 * size["pair_macs_per_site"] + 96 * size["block_outputs"]
                      + 5 * math.log2(V) * (size["block_outputs"] + 16 * len(ids)))
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------- exact
# baryon: quark string, diquark matrix (0: C gamma5; 1..3: eta_l C gamma_l), terms (coefficient, diquark pair, third)
_R2, _R6 = 1 / math.sqrt(2), 1 / math.sqrt(6)
_BARYON = {"p": ("udu", 0, [(1, 0, 1, 2)]), "n": ("udd", 0, [(-1, 0, 1, 2)]),
           "S+": ("usu", 0, [(-1, 0, 1, 2)]), "S-": ("dsd", 0, [(-1, 0, 1, 2)]),
           "X0": ("uss", 0, [(1, 0, 1, 2)]), "X-": ("dss", 0, [(-1, 0, 1, 2)]),
           "L": ("dsu", 0, [(_R6, 0, 1, 2), (_R6, 1, 2, 0), (-2 * _R6, 2, 0, 1)]),
           "S0": ("dsu", 0, [(_R2, 0, 1, 2), (-_R2, 1, 2, 0)]),
           "O1": ("sss", 1, [(1, 0, 1, 2)]), "O2": ("sss", 2, [(1, 0, 1, 2)]), "O3": ("sss", 3, [(1, 0, 1, 2)])}


@functools.lru_cache(maxsize=None)
def _channel_table():
    """Sink and source pairs of the ids 0..51 (octet) and 64..153 (decuplet)."""
    def cross(pairs, skip=()):
        return [(a, b) for a in pairs for b in pairs if (a, b) not in skip]
    sl, ll, ss = ("S0", "L"), ("L", "L"), ("S0", "S0")
    s2 = [ll, ("p", "X-"), ("n", "X0"), ("S+", "S-"), ss, sl]
    rows = [(("p", "n"), ("p", "n"))] + cross([("p", "L"), ("S+", "n"), ("S0", "p")])
    rows += cross(s2, {(ll, sl), (ss, sl), (sl, ll), (sl, ss)})
    rows += cross([("X-", "L"), ("S-", "X0"), ("S0", "X-")]) + [(("X-", "X0"), ("X-", "X0"))]
    table = dict(enumerate(rows))
    om = ("O1", "O2", "O3")
    pairs = list(itertools.product(om, om))
    table.update({64 + i: c for i, c in enumerate(itertools.product(pairs, pairs))})
    table.update({145 + i: (("p", a), ("p", b)) for i, (a, b) in enumerate(pairs)})
    return table


def _gamma(l):
    pauli = [np.array(m, dtype=complex) for m in ([[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]])]
    z = np.zeros((2, 2))
    g = [np.block([[z, -1j * s], [1j * s, z]]) for s in pauli] + [np.diag([1, 1, -1, -1]).astype(complex)]
    C = g[3] @ g[1]
    return (C @ g[0] @ g[1] @ g[2] @ g[3] if l == 0 else (1j, 1, -1j)[l - 1] * C @ g[l - 1]).real


@functools.lru_cache(maxsize=None)
def _tensor(name, ext):
    """Non-zero entries of the baryon tensor: quark indices [n, 3] and values [n]; ext: the free Dirac index."""
    _, l, terms = _BARYON[name]
    g, entries = _gamma(l), {}
    for coef, i, j, k in terms:
        for col in itertools.permutations(range(3)):
            sign = round(np.linalg.det(np.eye(3)[list(col)]))
            for ai, aj in zip(*np.nonzero(g)):
                spin = {i: int(ai), j: int(aj), k: ext}
                key = tuple(3 * spin[q] + col[q] for q in range(3))
                entries[key] = entries.get(key, 0.0) + coef * sign * g[ai, aj]
    return np.array(list(entries)), np.array(list(entries.values()))


def _sink(name, S, off, L):
    """U[eta0, eta1, eta2][a][site] as [1728, 2, V]: the sink tensor contracted with three propagators."""
    q = [S["s" if f == "s" else "l"] for f in _BARYON[name][0]]
    T = torch.zeros((2, 12, 12, 12), dtype=torch.float64, device="cuda")
    for a in range(2):
        idx, val = _tensor(name, off + a)
        T[(a,) + tuple(torch.as_tensor(i, device="cuda") for i in idx.T)] = torch.as_tensor(val, device="cuda")
    U = torch.empty((1728, 2, L ** 3), dtype=torch.complex128, device="cuda")
    for lo in range(0, L ** 3, 4096):
        x = slice(lo, lo + 4096)
        W = torch.einsum("aijk,vkn->vaijn", T.to(torch.complex128), q[2][x])
        W = torch.einsum("vaijn,vjm->vaimn", W, q[1][x])
        W = torch.einsum("vaimn,vil->lmnav", W, q[0][x])
        U[:, :, x] = W.reshape(1728, 2, -1)
    return U


def _fourier(U, L, inverse):
    for lo in range(0, U.shape[0], 216):
        part = U[lo:lo + 216].reshape(-1, L, L, L)
        f = torch.fft.ifftn if inverse else torch.fft.fftn
        U[lo:lo + 216] = f(part, dim=(1, 2, 3)).reshape(U[lo:lo + 216].shape)
    return U


@functools.lru_cache(maxsize=4096)
def _wick(sink_flavours, source, ap, bp):
    """Signed sum over the Wick contractions and both source tensors: sparse [i2][i1] (indices, values)."""
    (i3, w3), (i4, w4) = _tensor(source[0], ap), _tensor(source[1], bp)
    eta = np.concatenate([np.repeat(i3, len(i4), 0), np.tile(i4, (len(i3), 1))], 1)
    w = np.repeat(w3, len(w4)) * np.tile(w4, len(w3))
    src = _BARYON[source[0]][0] + _BARYON[source[1]][0]
    keys, vals = [], []
    for p in itertools.permutations(range(6)):
        if any(sink_flavours[i] != src[p[i]] for i in range(6)):
            continue
        sign = (-1) ** sum(p[i] > p[j] for i in range(6) for j in range(i + 1, 6))
        e = eta[:, list(p)]
        keys.append(((e[:, 3] * 12 + e[:, 4]) * 12 + e[:, 5]) * 1728 + (e[:, 0] * 12 + e[:, 1]) * 12 + e[:, 2])
        vals.append(sign * w)
    key, inv = np.unique(np.concatenate(keys), return_inverse=True)
    val = np.bincount(inv, np.concatenate(vals))
    keep = np.abs(val) > 1e-14
    return key[keep], val[keep]


def _exact_slice(ids, L, T, t0, t, Sl, Ss, lower, normalised):
    S = {"l": Sl.to(torch.complex128), "s": Ss.to(torch.complex128)}
    V, off = L ** 3, 2 if lower else 0
    table = _channel_table()
    out = torch.zeros((len(ids), V, 16), dtype=torch.complex128, device="cuda")
    by_sink = {}
    for n, i in enumerate(ids):
        by_sink.setdefault(table[i][0], []).append((n, table[i][1]))
    fields = {}
    for (b1, b2), members in by_sink.items():
        U1 = _fourier(_sink(b1, S, off, L), L, False)                 # B1 at q
        if b2 not in fields:
            fields = {b2: _fourier(_sink(b2, S, off, L), L, True)}    # B2 at -q, over V
        U2 = fields[b2]
        flavours = _BARYON[b1][0] + _BARYON[b2][0]
        flat = torch.view_as_real(U1).reshape(1728, -1)
        for n, source in members:
            for ap, bp in itertools.product(range(2), range(2)):
                key, val = _wick(flavours, source, off + ap, off + bp)
                if not len(key):
                    continue
                rows, inv = np.unique(key // 1728, return_inverse=True)
                W = torch.sparse_coo_tensor(np.stack([inv, key % 1728]), val, (len(rows), 1728), dtype=torch.float64,
                                            device="cuda").to_sparse_csr()
                rows = torch.as_tensor(rows, device="cuda")
                acc = torch.zeros((2, 2, V), dtype=torch.complex128, device="cuda")
                step = max(1, 2 ** 24 // V)
                WU = torch.view_as_complex((W @ flat).reshape(-1, 2, V, 2))
                for lo in range(0, len(rows), step):
                    acc += torch.einsum("rav,rbv->bav", WU[lo:lo + step], U2[rows[lo:lo + step]])
                c = torch.fft.ifftn(acc.reshape(4, L, L, L), dim=(1, 2, 3)) * V
                lo = 4 * ap + 8 * bp
                out[n, :, lo:lo + 4] = c.reshape(4, V).T
        if normalised:
            strange = flavours.count("s")
            f = math.exp(((6 - strange) * M_UD + strange * M_S) * _distance(t, t0, T, lower))
            for n, _ in members:
                out[n] *= f
    return out


def exact(case, seed):
    ids, dtype = _ids(case["channels"]), DTYPE[case["dtype"]]
    if case["kind"] == "project":
        return _exact_projection(case["L"], _correlators(case, seed))
    if not set(ids) <= set(_channel_table()):
        return None
    if case["kind"] == "batch":
        if max(L for L, _ in _lattices(case)) > 24:
            return None
        outs, k = [], case["sources"]
        for L, T in _lattices(case):
            Sl, Ss = _propagators(seed, L, T, 0, range(T), case["field"], dtype)
            outs.append(_exact_slice(ids, L, T, (k - 1) * T // k, T - 1, Sl[-1], Ss[-1], False, True))
        return outs
    # a few seconds at most; 48^3 would take longer
    if case["L"] ** 3 * case["slices"] > 2 * 32 ** 3:
        return None
    times = list(range(case["T"])) if case["kind"] == "stream" else _times(case)
    Sl, Ss = _propagators(seed, case["L"], case["T"], case["t0"], times, case["field"], dtype, case["lower"])
    assert len(set(times)) == len(times)  # a slice is found by its time below
    return torch.stack([_exact_slice(ids, case["L"], case["T"], case["t0"], t, Sl[times.index(t)], Ss[times.index(t)],
                                     case["lower"], case["normalised"]) for t in _times(case)])


def _exact_projection(L, C):
    """Source spin states (0,0), (1,1), (1,0), (1,-1) and their mean over the 24 rotations of the cube."""
    v = C.reshape(C.shape[:-1] + (4, 4))  # [p = a' + 2 b', a + 2 b]
    R = torch.stack([(v[..., 2, :] - v[..., 1, :]) * _R2, v[..., 0, :], (v[..., 2, :] + v[..., 1, :]) * _R2,
                     v[..., 3, :]], dim=-2).reshape(C.shape)
    r = np.arange(L ** 3)
    r = np.stack([r % L, r // L % L, r // L ** 2])
    A = torch.zeros_like(R)
    for perm in itertools.permutations(range(3)):
        for signs in itertools.product((1, -1), repeat=3):
            M = np.diag(signs) @ np.eye(3, dtype=int)[list(perm)]
            if round(np.linalg.det(M)) == 1:
                x = M @ r % L
                A += R[..., torch.as_tensor(x[0] + L * (x[1] + L * x[2]), device="cuda"), :]
    return [R, A / 24]
