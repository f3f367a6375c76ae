"""Performance cases: the work a user of this library has it do, through the public binding.

Each case names a kind of call and its sizes; `prepare` makes what the user's program holds before the call,
`run` makes one call (or the short sequence of calls that belongs together) and returns everything it computes.

Molecules are the seeded water clusters of this repository, 1 to 24 waters (50 to 1200 basis functions, 137
auxiliary functions a water, 5 occupied orbitals a water). `cut` leaves out the last `cut` hydrogens and makes up
for their electrons with the charge, so that sizes are not all multiples of 50.
"""
import numpy as np
import torch

from paper_1707_03771_gb300 import binding, clusters

FP64, SPLIT = "fp64", "split"


def listed():
    return [
        # one J/K build of the smallest cluster through host arrays: a program that drives its own SCF on a
        # small molecule; the call's latency and its launches are what it waits for
        {"name": "jk_fp64_2", "kind": "jk", "waters": 2, "cut": 0, "precision": FP64, "slices": 0, "host": True},
        # an FP64 J/K build of an ordinary molecule
        {"name": "jk_fp64_8", "kind": "jk", "waters": 8, "cut": 0, "precision": FP64, "slices": 0, "host": False},
        # the early iterations of a split-precision SCF build the exchange from 3 slices; a ragged size
        {"name": "jk_split3_12", "kind": "jk", "waters": 12, "cut": 1, "precision": SPLIT, "slices": 3, "host": False},
        # the late iterations build it from 5 slices: an ordinary and the largest cluster. At 24 waters a handle
        # with its slices takes about 80 GB (the 32-water workload takes 180 GB, and several handles share the GPU)
        {"name": "jk_split5_16", "kind": "jk", "waters": 16, "cut": 0, "precision": SPLIT, "slices": 5, "host": False},
        {"name": "jk_split5_24", "kind": "jk", "waters": 24, "cut": 0, "precision": SPLIT, "slices": 5, "host": False},
        # a new geometry: integrals, metric factor and whitening, then its first J/K build (which cuts B's
        # slices in split precision). A geometry optimisation does this once a step.
        {"name": "build_fp64_4", "kind": "build", "waters": 4, "cut": 0, "precision": FP64, "slices": 0},
        {"name": "build_split_12", "kind": "build", "waters": 12, "cut": 0, "precision": SPLIT, "slices": 5},
        # whole calls: a small molecule from its geometry to converged FP64 results, and the first iterations of
        # a split-precision SCF from the superposition of atomic densities on a handle that has its B
        {"name": "scf_fp64_2", "kind": "molecule", "waters": 2, "cut": 0},
        {"name": "scf_split_8", "kind": "scf", "waters": 8, "cut": 0, "iterations": 8},
        # the correlation energy after an SCF
        {"name": "mp2_4", "kind": "mp2", "waters": 4, "cut": 0},
        # the density-fitting object operations: half transformation, exchange, density fit and Coulomb matrix
        # of one object, as a program writes its own method with them
        {"name": "ops_4", "kind": "ops", "naux": 548, "n": 200, "nocc": 20},
        # the learned guess: training epochs of the network of the diagonal water blocks on a small training set
        {"name": "train_281", "kind": "train", "samples": 281, "nin": 57, "nout": 1275, "batch": 16, "epochs": 4},
    ]


def _spread(rng, lo, hi):
    """A whole number, uniform over the logarithm of [lo, hi]."""
    return min(hi, max(lo, round(lo * (hi / lo) ** rng.random())))


def draw(rng):
    known = [{k: v for k, v in c.items() if k != "name"} for c in listed()]
    while True:
        case = _draw(rng)
        if case not in known:
            return case


def _draw(rng):
    kind = rng.choice(["jk", "jk", "jk", "jk", "build", "build", "molecule", "scf", "mp2", "ops", "train"])
    cut = rng.choice([0, 0, 1, 2])
    if kind == "jk":
        precision = rng.choice([FP64, SPLIT, SPLIT])
        return {"kind": "jk", "waters": _spread(rng, 1, 9 if precision == FP64 else 23), "cut": cut,
                "precision": precision, "slices": 0 if precision == FP64 else rng.choice([3, 5]),
                "host": rng.random() < 0.5}
    if kind == "build":
        precision = rng.choice([FP64, SPLIT])
        return {"kind": "build", "waters": _spread(rng, 1, 5 if precision == FP64 else 14), "cut": cut,
                "precision": precision, "slices": 0 if precision == FP64 else 5}
    if kind == "molecule":      # water clusters, or with a hydroxide ion in them
        return {"kind": "molecule", "waters": rng.choice([1, 2, 3]), "cut": rng.choice([0, 1])}
    if kind == "scf":
        return {"kind": "scf", "waters": _spread(rng, 2, 12), "cut": 0, "iterations": rng.randint(4, 8)}
    if kind == "mp2":
        return {"kind": "mp2", "waters": _spread(rng, 1, 6), "cut": cut}
    if kind == "ops":
        n = _spread(rng, 23, 260)
        return {"kind": "ops", "naux": _spread(rng, 37, 700), "n": n, "nocc": max(1, n // rng.choice([5, 7, 10]))}
    if rng.random() < 0.5:      # the network of the pair blocks, or of the diagonal blocks
        return {"kind": "train", "samples": _spread(rng, 64, 900), "nin": 26, "nout": 2500, "batch": 64,
                "epochs": rng.randint(1, 4)}
    return {"kind": "train", "samples": _spread(rng, 32, 400), "nin": 57, "nout": 1275, "batch": 16,
            "epochs": rng.randint(1, 4)}


def _system(case, seed):
    """A water cluster of the case's size (another seed, another geometry) without its last `cut` hydrogens."""
    full = clusters.water_cluster(case["waters"], 1000 + seed % 1000003)
    cut = case["cut"]
    if cut == 0:
        return full
    atoms = full.atoms[:len(full.atoms) - cut]
    # an even electron count: each missing H took its electron along, the charge gives or takes one
    return clusters.make_system(atoms, charge=-(cut % 2), label=full.label + f"-{cut}H")


def _sizes(case):
    n = 50 * case["waters"] - 10 * case["cut"]
    naux = 137 * case["waters"] - 25 * case["cut"]
    nocc = (10 * case["waters"] - case["cut"] + case["cut"] % 2) // 2
    return n, naux, nocc


def _orbitals(n, nocc, rng):
    """Orthonormal occupied orbitals that each sit mainly on one block of about 50 functions, as localised
    occupied orbitals sit on one water, with tails everywhere."""
    C = 0.03 * rng.standard_normal((n, nocc))
    for i in range(nocc):
        b = min(50 * (i // 5), max(0, n - 50))
        C[b:b + 50, i] += rng.standard_normal(min(50, n))
    return np.linalg.qr(C)[0]


def _precision(case):
    return binding.DF_PREC_FP64 if case["precision"] == FP64 else binding.DF_PREC_SPLIT


def _jk_inputs(state, handle, rng):
    C = _orbitals(handle.n, handle.nocc, rng)
    D = 2.0 * C @ C.T
    state.update(D=D, C=C)
    if not state["case"].get("host", False):
        state["dD"], state["dC"] = torch.from_numpy(D).cuda(), torch.from_numpy(np.ascontiguousarray(C)).cuda()
        state["dJ"], state["dK"] = torch.empty_like(state["dD"]), torch.empty_like(state["dD"])


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    state = {"case": case}
    if kind in ("jk", "build", "scf", "mp2"):
        # the molecule's handle; calls other than "build" find its B built, as a user's program keeps it
        h = state["handle"] = binding.Handle(_system(case, seed))
        if kind != "build":
            h.build_B()
        if kind in ("jk", "build"):
            _jk_inputs(state, h, rng)
        if kind == "mp2":
            # orthonormal orbitals and ascending energies with a gap (core, valence, virtual)
            n, no = h.n, h.nocc
            state["C"] = np.linalg.qr(np.hstack([_orbitals(n, no, rng), rng.standard_normal((n, n - no))]))[0]
            state["eps"] = np.concatenate([np.sort(rng.uniform(-1.4, -0.45, no)), np.sort(rng.gamma(1.2, 4.0, n - no) + 0.1)])
            state["eps"][:max(1, no // 5)] = -20.5
    elif kind == "molecule":
        state["system"] = _system(case, seed)
    elif kind == "ops":
        naux, n, no = case["naux"], case["n"], case["nocc"]
        # the tensor operations need a handle for their device and stream: a water's
        h = state["handle"] = binding.Handle(clusters.water_cluster(1, 5))
        T, C, D = _ops_inputs(case, seed)
        state.update(T=binding.DFTensor.create(h, T), C=C, D=D)
    elif kind == "train":
        state["net"] = binding.Mlp(case["nin"], 256, 3, case["nout"], seed=seed % 1000)
        state["p0"] = state["net"].params()
        # features: radial histograms and coordinates of neighbours; targets: a mean block and its variation
        X = np.abs(rng.standard_normal((case["samples"], case["nin"]))) * rng.uniform(0.1, 1.5, case["nin"])
        Y = 0.3 * rng.standard_normal(case["nout"]) + 0.05 * np.tanh(X @ rng.standard_normal((case["nin"], case["nout"])))
        state.update(X=X.astype(np.float32), Y=Y.astype(np.float32))
    return state


def _ops_inputs(case, seed):
    """A fitted object (symmetric in its orbital indices, decaying along the auxiliary index and away from the
    diagonal), occupied orbitals and their density."""
    rng = np.random.default_rng(seed)
    naux, n, no = case["naux"], case["n"], case["nocc"]
    i = np.arange(n)
    decay = np.exp(-np.abs(i[:, None] - i[None, :]) / 40.0)
    T = rng.standard_normal((naux, n, n)) * (0.05 + np.exp(-np.arange(naux) / 150.0))[:, None, None]
    T = 0.5 * (T + T.transpose(0, 2, 1)) * decay
    C = _orbitals(n, no, rng)
    return np.ascontiguousarray(T), np.ascontiguousarray(C), 2.0 * C @ C.T


def _jk(state):
    case, h = state["case"], state["handle"]
    if case.get("host", False):
        J, K = h.jk(state["D"], state["C"], _precision(case), case["slices"] or 3)
        return {"J": J, "K": K}
    h.jk_device(state["dD"].data_ptr(), state["dC"].data_ptr(), state["C"].shape[1], state["dJ"].data_ptr(),
                state["dK"].data_ptr(), _precision(case), case["slices"] or 3)
    return {"J": state["dJ"], "K": state["dK"]}


def _results(h, r):
    """What a user reads after an SCF: the energy and its parts, the density, the Fock matrix."""
    return {"energy": r["energy"], "one": r["e_one"], "coulomb": r["e_coul"], "exchange": r["e_exch"],
            "D": h.matrix("D"), "F": h.matrix("F")}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "jk":
        return _jk(state)
    h = state.get("handle")
    if kind == "build":
        h.build_B(whitening=binding.DF_WHITEN_FP64 if case["precision"] == FP64 else binding.DF_WHITEN_SPLIT)
        return _jk(state)
    if kind == "molecule":
        # converged well below the default thresholds: the density is then determined to the bound of its type
        with binding.Handle(state["system"]) as fresh:
            r = fresh.scf(conv_E=1e-11, conv_err=1e-9)
            return _results(fresh, r)
    if kind == "scf":
        # a fixed number of iterations: where the last bits of the convergence test fall must not decide how
        # many are timed
        r = h.scf(max_iter=case["iterations"], conv_E=1e-14, precision=binding.DF_PREC_SPLIT, slices=3, incremental=1,
                  approx_diag=1, guess="sad")
        return _results(h, r)
    if kind == "mp2":
        return {"e2": h.mp2(state["C"], state["eps"])}
    if kind == "ops":
        T = state["T"]
        Y = T.transform("first", state["C"])
        K = Y.contract(Y, "first")
        Y.close()
        g = T.density_fit(state["D"])
        return {"K": K, "fit": g, "J": T.density_back(g)}
    state["net"].set_params(state["p0"])
    hist = state["net"].train(state["X"], state["Y"], case["epochs"], case["batch"], 3e-4, seed=3)
    return {"loss": hist, "params": state["net"].params()}


def work(case):
    kind = case["kind"]
    if kind == "ops":
        naux, n, no = case["naux"], case["n"], case["nocc"]
        return {"bytes": 8.0 * (naux * n * n + n * no + 3 * n * n + naux),
                "flops": 2.0 * naux * n * n * no + 1.0 * naux * no * n * (n + 1) + 4.0 * naux * n * n}
    if kind == "train":
        w = case["nin"] * 256 + 2 * 256 * 256 + 256 * case["nout"]
        steps = case["epochs"] * (case["samples"] // min(case["batch"], case["samples"]))
        rows = min(case["batch"], case["samples"])
        # per step: forward, weight gradients and (but for the first layer) input gradients
        return {"bytes": 4.0 * (2 * w + case["samples"] * (case["nin"] + case["nout"])),
                "flops": steps * rows * 2.0 * (3 * w - case["nin"] * 256)}
    n, naux, nocc = _sizes(case)
    pairs = n * (n + 1) // 2
    matrices = 8.0 * (3 * n * n + n * nocc)                 # D, C, J, K
    coulomb = 4.0 * naux * pairs
    exchange = 2.0 * naux * n * n * nocc + 1.0 * naux * n * (n + 1) * nocc
    b = 8.0 * naux * pairs                                  # B, packed by symmetry
    fit = naux ** 3 / 3.0 + 1.0 * naux * naux * pairs       # metric factor, triangular whitening
    if kind == "jk":
        return {"bytes": b + matrices, "flops": coulomb + exchange}
    if kind == "build":
        return {"bytes": b + matrices, "flops": fit + coulomb + exchange}
    if kind == "mp2":
        nv = n - nocc
        return {"bytes": b + 8.0 * (n * n + n),
                "flops": 2.0 * naux * nocc * (n * n + n * nv) + 1.0 * naux * (nocc * nv) * (nocc * nv + 1)}
    algebra = 2.0 * (3.0 * n ** 3 + 2.0 * n * n * nocc) + 9.0 * n ** 3     # products and the eigensolve
    iterations = case.get("iterations", 14)
    one = {"bytes": iterations * b + matrices, "flops": iterations * (coulomb + exchange + algebra)}
    if kind == "molecule":
        one["flops"] += fit
    return one


def exact(case, seed):
    """64-bit results of plain numpy for the tensor operations, whose inputs are all given. The other kinds start
    from integrals over the basis (which only this library's own code gives) or, in training, from batches
    that the library's generator shuffles: their results have no value that plain numpy gives from the
    case's inputs alone."""
    if case["kind"] != "ops":
        return None
    T, C, D = _ops_inputs(case, seed)
    naux, n, _ = T.shape
    Y = np.matmul(C.T[None], T).reshape(-1, n)              # (naux nocc) x n
    g = T.reshape(naux, -1) @ D.reshape(-1)
    return {"K": Y.T @ Y, "fit": g, "J": (g @ T.reshape(naux, -1)).reshape(n, n)}
