"""The work that programs built on the hop engine have it do, for timing.

A case is a dict of plain values; prepare() builds what a program holds before
the call (a populated lattice, or the description of a simulation), run() is one
pass through the public entry points, and returns the counts and the positions
that the program reads.  Every output is a whole number that follows from the
seed alone, whatever the launch shapes are.  Simulations without reactions read the
unwrapped positions of their walkers; those with reactions, whose molecules change
in number, save the whole occupancy grid.
"""
import math

import numpy as np

import paper_1605_03726_gb300 as psc

RV = 1e-8
AB_D, AB_K = 1e-12, 1e-19                   # A + B -> C: D of A and B, rate constant
AB_TAU = 2 * RV * RV / (3 * AB_D)           # hop interval of A and B


def listed():
    return [
        # a small box of walkers, followed step by step: the shortest calls
        dict(name="diffuse_64", kind="diffuse", ni=64, nj=64, nk=64, flags=7, D=1e-11, occ=0.01, D2=0.0, occ2=0.0,
             crowd=0.0, steps=1, events=100),
        # A + B -> C with immobile C, one whole simulation of 1000 hop intervals from creation to the final grid
        dict(name="ab_64", kind="ab", ni=64, nj=64, nk=64, flags=7, n_a=2000, n_b=2000, taus=1000),
        # an enzymatic cascade of 22 species and 30 reactions: many short lists, events of unrelated periods
        dict(name="mapk_200", kind="mapk", ni=200, nj=200, nk=200, flags=7, model=5, scale=1.0, steps=4, events=500),
        # a round cell: ligands in the cytoplasm bind receptors in the membrane, walkers outside
        dict(name="cell_128", kind="cell", ni=128, nj=128, nk=128, flags=7, radius=100.0, ligands=30000,
             receptors=5000, outside=10000, steps=4, events=250),
        # the paper's OpenMP workload: 160^3 at 30 % occupancy
        dict(name="dense_160", kind="diffuse", ni=160, nj=160, nk=160, flags=7, D=1e-12, occ=0.30, D2=0.0, occ2=0.0,
             crowd=0.0, steps=1, events=100),
        # the FCC lattice (ABC stacking) at 10 %
        dict(name="fcc_192", kind="diffuse", ni=192, nj=192, nk=192, flags=15, D=1e-11, occ=0.10, D2=0.0, occ2=0.0,
             crowd=0.0, steps=1, events=100),
        # two walker species of different hop intervals among immobile crowders: their events alternate
        dict(name="walkers_256", kind="diffuse", ni=256, nj=256, nk=256, flags=7, D=1e-11, occ=0.03, D2=7e-12,
             occ2=0.02, crowd=0.20, steps=1, events=100),
        # a closed box of odd sizes
        dict(name="ragged_300", kind="diffuse", ni=301, nj=251, nk=211, flags=0, D=1e-11, occ=0.05, D2=0.0, occ2=0.0,
             crowd=0.0, steps=1, events=100),
        # reversible A + B <-> C under 30 % crowding behind reflective walls
        dict(name="crowded_256", kind="crowded", ni=256, nj=256, nk=256, flags=0, crowd=0.30, fa=0.05, fb=0.01,
             steps=4, events=100),
        # the headline lattice: 512^3 at 1 %, counts after every 100 events
        dict(name="diffuse_512", kind="diffuse", ni=512, nj=512, nk=512, flags=7, D=1e-11, occ=0.01, D2=0.0, occ2=0.0,
             crowd=0.0, steps=5, events=100),
        # the largest lattices a program sets up on one device
        dict(name="diffuse_1024", kind="diffuse", ni=1024, nj=1024, nk=1024, flags=7, D=1e-11, occ=0.01, D2=0.0,
             occ2=0.0, crowd=0.0, steps=1, events=50),
        # a parameter sweep: replicas of the A + B -> C model, edges 32-160, 1-20 %, through the batching server
        dict(name="serve_64", kind="serve", replicas=64, lo=32, hi=160, taus=250),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _edges(rng, lo, hi, fcc, spread=1.6):
    """Three extents around one size, and boundary flags that fit them (odd sizes along closed axes)."""
    e = _log(rng, lo, hi)
    n = [max(8, int(min(hi * 1.2, e * _log(rng, 1 / spread, spread)))) for _ in range(3)]
    flags = 7 if rng.random() < 0.6 else rng.randrange(8)
    if flags & 2:
        n[1] += n[1] & 1
    if flags & 4:
        n[2] += (-n[2]) % (6 if fcc else 2)
    if rng.random() < 0.5:                  # half of the lattices have round extents
        n = [(x + 7) // 8 * 8 for x in n]
        if fcc:
            n[2] = (n[2] + 23) // 24 * 24
    return n, flags | (8 if fcc else 0)


def draw(rng):
    kind = rng.choice(["diffuse", "diffuse", "diffuse", "fcc", "walkers", "ab", "mapk", "cell", "crowded", "serve"])
    if kind in ("diffuse", "fcc", "walkers"):
        (ni, nj, nk), flags = _edges(rng, 32, 900 if kind == "diffuse" else 320, kind == "fcc")
        V = ni * nj * nk
        two = kind == "walkers"
        occ = min(_log(rng, 0.005, 0.4), 1e7 / V)
        occ2 = min(_log(rng, 0.005, 0.2), 5e6 / V) if two else 0.0
        n = V * (occ + occ2)
        return dict(kind="diffuse", ni=ni, nj=nj, nk=nk, flags=flags, D=_log(rng, 1e-12, 1e-11), occ=occ,
                    D2=_log(rng, 1e-12, 1e-11) if two else 0.0, occ2=occ2,
                    crowd=rng.choice([0.0, 0.1, 0.3]) if two else 0.0, steps=rng.choice([1, 2]),
                    events=int(min(rng.randint(30, 120), max(10, 1.5e8 / n))))
    if kind == "ab":
        (ni, nj, nk), flags = _edges(rng, 32, 112, False)
        n = int(ni * nj * nk * _log(rng, 0.004, 0.04))
        return dict(kind="ab", ni=ni, nj=nj, nk=nk, flags=flags, n_a=n, n_b=int(n * rng.uniform(0.5, 1.5)),
                    taus=rng.randint(200, 1000))
    if kind == "mapk":
        (ni, nj, nk), flags = _edges(rng, 100, 240, False, 1.2)
        return dict(kind="mapk", ni=ni, nj=nj, nk=nk, flags=flags, model=rng.randrange(1000),
                    scale=_log(rng, 0.1, 2.0), steps=rng.randint(2, 4), events=rng.randint(100, 300))
    if kind == "cell":
        e = rng.randint(36, 90) * 2
        r = rng.uniform(0.55, 0.78) * e
        room = 4.19 * r ** 3 / (2 * 1.73 * 1.63)
        return dict(kind="cell", ni=e, nj=e, nk=e, flags=7, radius=r, ligands=int(room * _log(rng, 0.002, 0.05)),
                    receptors=int(r * r * _log(rng, 0.05, 0.4)), outside=int(e ** 3 * _log(rng, 0.001, 0.02)),
                    steps=rng.randint(1, 3), events=rng.randint(100, 300))
    if kind == "crowded":
        (ni, nj, nk), flags = _edges(rng, 64, 256, False, 1.2)
        return dict(kind="crowded", ni=ni, nj=nj, nk=nk, flags=flags, crowd=rng.uniform(0.0, 0.4),
                    fa=_log(rng, 0.005, 0.06), fb=_log(rng, 0.002, 0.02), steps=rng.randint(1, 2),
                    events=rng.randint(40, 120))
    return dict(kind="serve", replicas=rng.randint(16, 96), lo=32, hi=rng.randint(64, 140), taus=rng.randint(100, 250))


# ---------------------------------------------------------------------------
# models
# ---------------------------------------------------------------------------
def _n(case):
    V = case["ni"] * case["nj"] * case["nk"]
    return int(V * case["occ"]), int(V * case["occ2"]), int(V * case["crowd"])


def _mapk_model(case):
    """Species (D, count) and reactions of a dual-phosphorylation cascade of three tiers: ten steps
    E + S <-> ES -> E + P; counts, D and rates drawn from the case's model number."""
    rnd = np.random.RandomState(case["model"])
    logu = lambda lo, hi: float(math.exp(rnd.uniform(math.log(lo), math.log(hi))))
    names, species, reactions = {}, [], []

    def add(name, count):
        names[name] = len(species)
        species.append((logu(0.5e-12, 10e-12), int(count * case["scale"])))

    for name in ("E1", "E2", "KKPase", "KPase"):
        add(name, rnd.randint(50, 500))
    for name in ("KKK", "KK", "K"):
        add(name, rnd.randint(1000, 20000))
    for name in ("KKK*", "KKp", "KKpp", "Kp", "Kpp"):
        add(name, 0)
    for e, s, p in [("E1", "KKK", "KKK*"), ("E2", "KKK*", "KKK"), ("KKK*", "KK", "KKp"), ("KKK*", "KKp", "KKpp"),
                    ("KKPase", "KKpp", "KKp"), ("KKPase", "KKp", "KK"), ("KKpp", "K", "Kp"), ("KKpp", "Kp", "Kpp"),
                    ("KPase", "Kpp", "Kp"), ("KPase", "Kp", "K")]:
        add(e + ":" + s, 0)
        es = names[e + ":" + s]
        reactions.append(([names[e], names[s]], [es], logu(1e-20, 1e-18)))
        reactions.append(([es], [names[e], names[s]], logu(0.1, 100.0)))
        reactions.append(([es], [names[e], names[p]], logu(0.1, 100.0)))
    return species, reactions


def _cell_labels(case):
    """0 outside, 1 a membrane shell 1.5 voxel radii thick, 2 the cytoplasm of a round cell."""
    x = [s * (np.arange(n) - (n - 1) / 2.0) for s, n in ((2.0, case["ni"]), (1.73, case["nj"]), (1.63, case["nk"]))]
    r = np.sqrt(x[2][:, None, None] ** 2 + x[1][None, :, None] ** 2 + x[0][None, None, :] ** 2)
    return ((r < case["radius"]).astype(np.uint8) + (r < case["radius"] - 1.5)).astype(np.uint8)


def _lattice(case):
    return psc.Lattice(case["ni"], case["nj"], case["nk"], voxel_radius=RV, boundary=case["flags"])


def _replicas(case, seed):
    rnd = np.random.RandomState(seed)
    out = []
    for r in range(case["replicas"]):
        e = 2 * rnd.randint(case["lo"] // 2, case["hi"] // 2 + 1)
        half = int(rnd.uniform(0.01, 0.20) * e ** 3 / 2)
        out.append(((e, e, e), [half, half, 0], int(seed) * 1000 + r))
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "ab":
        return dict(case=case, seed=seed)
    if kind == "serve":
        return dict(case=case, replicas=_replicas(case, seed))
    L = _lattice(case)
    walkers = []
    if kind == "diffuse":
        n, n2, crowd = _n(case)
        if crowd:
            L.add_species(0.0, crowd)
        walkers.append(L.add_species(case["D"], n))
        if n2:
            walkers.append(L.add_species(case["D2"], n2))
    elif kind == "mapk":
        species, reactions = _mapk_model(case)
        for D, n in species:
            L.add_species(D, n)
        for re, pr, k in reactions:
            L.add_reaction(re, pr, k)
    elif kind == "cell":
        L.set_compartments(_cell_labels(case), 3)
        lig = L.add_species(1e-12, case["ligands"], compartment=2)
        rec = L.add_species(0.1e-12, case["receptors"], compartment=1)
        lr = L.add_species(0.05e-12, 0, compartment=1)
        L.add_species(1e-12, case["outside"], compartment=0)
        L.add_reaction([lig, rec], [lr], 5e-19)
        L.add_reaction([lr], [rec, lig], 20.0)
    else:
        V = case["ni"] * case["nj"] * case["nk"]
        if case["crowd"] > 0:
            L.add_species(0.0, int(case["crowd"] * V))
        a = L.add_species(5e-12, int(case["fa"] * V))
        b = L.add_species(1e-12, int(case["fb"] * V))
        c = L.add_species(0.5e-12, 0)
        L.add_reaction([a, b], [c], 1e-19)
        L.add_reaction([c], [a, b], 10.0)
    L.populate(seed)
    return dict(case=case, L=L, walkers=walkers)


def _snapshot(L):
    return L.grid().view(np.int16)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "ab":
        with _lattice(case) as L:
            a, b, c = L.add_species(AB_D, case["n_a"]), L.add_species(AB_D, case["n_b"]), L.add_species(0.0, 0)
            L.add_reaction([a, b], [c], AB_K)
            L.populate(state["seed"])
            L.run(case["taus"] * AB_TAU)
            return [L.counts(), _snapshot(L)]
    if kind == "serve":
        S = psc.Server(max_device_bytes=32 << 30, max_active=512)
        tickets = [S.submit(shape, [AB_D, AB_D, 0.0], counts, [((0, 1), (2,), AB_K)], seed, case["taus"] * AB_TAU)
                   for shape, counts, seed in state["replicas"]]
        while S.step(64) != (0, 0):
            pass
        counts = np.stack([S.result(t)[0] for t in tickets])
        S.close()
        return counts
    L = state["L"]
    counts = []
    for _ in range(case["steps"]):
        L.run_events(case["events"])
        counts.append(L.counts())
    if kind != "diffuse":
        return [np.stack(counts), _snapshot(L)]
    out = [np.stack(counts)]
    for s in state["walkers"]:
        xyz, ids = L.unwrapped(s)
        out += [xyz, ids.view(np.int32)]
    return out


def work(case):
    """Per attempt (a molecule in one event of its species): its voxel (4 bytes), the target's occupancy (2), the
    claim written and read back (8) and, for the hops that succeed, the voxel (4) and both occupancies (4) written;
    about 400 operations of the draw, the neighbour and the claim.  Read-out: 16 bytes for each walker, 2 for each
    voxel of a grid."""
    kind = case["kind"]
    events = case.get("steps", 1) * case.get("events", 0)
    V = case["ni"] * case["nj"] * case["nk"] if "ni" in case else 0
    out = 2.0 * V
    if kind == "diffuse":
        n, n2, crowd = _n(case)
        free = 1.0 - (n + n2 + crowd) / V
        attempts = events * (n * case["D"] + n2 * case["D2"]) / (case["D"] + case["D2"])
        out = 16.0 * (n + n2)
    elif kind == "ab":
        free = 0.98
        attempts = 0.5 * case["taus"] * (case["n_a"] + case["n_b"])     # the counts fall as C forms
    elif kind == "serve":
        mid = sum(float(e) ** 3 for e in range(case["lo"], case["hi"] + 1, 2)) / ((case["hi"] - case["lo"]) // 2 + 1)
        free, attempts = 0.9, 0.4 * case["taus"] * case["replicas"] * mid * 0.105
    elif kind == "mapk":
        species, _ = _mapk_model(case)
        free, attempts = 0.99, events * sum(D * n for D, n in species) / sum(D for D, _ in species)
    elif kind == "cell":
        free = 0.9
        attempts = events * (case["ligands"] + 0.1 * case["receptors"] + case["outside"]) / 2.15
    else:
        free = 1.0 - case["crowd"] - case["fa"] - case["fb"]
        attempts = events * V * (5.0 * case["fa"] + case["fb"]) / 6.5
    return {"bytes": float(attempts * (14.0 + 8.0 * free) + out), "flops": float(400.0 * attempts)}


def exact(case, seed):
    """The outputs are whole numbers, decided by 32-bit draws: nothing is rounded, they are equal or wrong."""
    return None
