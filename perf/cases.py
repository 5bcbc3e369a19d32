"""Workloads of the library: what its users run, through its public entry points.

listed() names the workloads, draw() gives more of the same ranges, prepare()
builds what a program holds before the call (the contexts with their orders, the
couplings), run() is one pass, work() its floor and exact() the same results in
64-bit torch arithmetic.  Sizes come from the repository's workload
configurations (square lattices of side 6 to 24, mixed batches of side 8 to 20,
chimera cells, cubic lattices, 3-regular graphs of up to 200 spins, Max-2-SAT,
3-state Potts lattices) and from the max-plus GEMM's step shapes.

Energies of FP32 contexts are float32 results that the entry points hand over as
doubles; run() returns them as float32.  Counts are returned as 64-bit limbs.
"""
import numpy as np
import torch

import instances as I
import paper_2008_06888_gb300 as P
from paper_2008_06888_gb300 import binding as B

# ---------------------------------------------------------------- the cases


def listed():
    return [
        # the smallest call: one small lattice at a time, energy and exact count
        # (36 spins, row by row); launches and host latency are all of it
        dict(name="single_square6", kind="single", L=6),
        # the headline workload: ground states of 24 x 24 Gaussian lattices with
        # fields along one greedy order, a batch of coupling sets on the device
        dict(name="config_square24", kind="config", L=24, W=24, B=16, restarts=64),
        # many disorder instances of uneven size with exact counts in one call
        dict(name="mixed_counts", kind="mixed", B=192, Lmin=8, Lmax=20),
        # hardware-graph instances (K_{4,4} cells): energy and exact count of one
        dict(name="chimera6_count", kind="chimera", L=6),
        # optimal assignments of Max-2-SAT formulas on one graph: minimum of
        # violated clauses and exact count of optimal assignments
        dict(name="max2sat140_counts", kind="max2sat", N=140, B=16, graph=500),
        # random 3-regular glass, N = 200: the order needs max-plus GEMM steps
        # and transposes; ground states by traceback
        dict(name="rrg200_config", kind="rrg", N=200, B=4, graph=3),
        # 3-state Potts glass (q = 3), an odd side; ground state by traceback
        dict(name="potts15_config", kind="potts", L=15, B=1),
        # the 3D workload: ground states of open cubic lattices
        dict(name="cubic5x5x6_config", kind="cubic", L=6, W=5, H=5, B=4),
        # uniform samples of all ground states of a degenerate lattice: a chain
        # of small batched counts
        dict(name="sample_square12", kind="sample", L=12, samples=16),
        # max-plus product of the pairwise steps, square and large, float32
        dict(name="gemm_f32_2048", kind="gemm", dtype="f32", batch=2, M=2048, N=2048, K=2048,
             ta=0, tb=0),
        # the same in integers, ragged sizes and a transposed operand
        dict(name="gemm_i32_ragged", kind="gemm", dtype="i32", batch=5, M=777, N=1001, K=333,
             ta=1, tb=0),
        # gradient-based use: E(J, h) and its gradient (the ground state) of one
        # lattice through autograd, row-by-row order
        dict(name="autograd_square18", kind="autograd", L=18),
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    # chimera lattices come in few sizes: drawn half as often as the others
    kind = rng.choice(["single", "config", "mixed", "max2sat", "rrg", "potts", "cubic", "sample",
                       "gemm", "autograd"] * 2 + ["gemm", "chimera"])
    if kind == "single":
        return dict(kind=kind, L=rng.randint(5, 14))
    if kind == "config":
        return dict(kind=kind, L=rng.randint(12, 24), W=rng.randint(12, 24),
                    B=rng.randint(1, 16), restarts=32)
    if kind == "mixed":
        lo = rng.randint(6, 16)
        return dict(kind=kind, B=_log(rng, 12, 192), Lmin=lo, Lmax=rng.randint(lo, 20))
    if kind == "chimera":
        return dict(kind=kind, L=rng.randint(3, 5))
    if kind == "max2sat":
        return dict(kind=kind, N=2 * rng.randint(25, 70), B=rng.randint(1, 16),
                    graph=rng.randint(1, 400))
    if kind == "rrg":
        return dict(kind=kind, N=2 * rng.randint(40, 80), B=rng.randint(1, 4),
                    graph=rng.randint(1, 400))
    if kind == "potts":
        return dict(kind=kind, L=rng.randint(5, 14), B=rng.randint(1, 3))
    if kind == "cubic":
        return dict(kind=kind, L=rng.randint(4, 6), W=rng.randint(3, 5), H=rng.randint(3, 5),
                    B=rng.randint(1, 4))
    if kind == "sample":
        return dict(kind=kind, L=rng.randint(5, 12), samples=rng.randint(1, 16))
    if kind == "gemm":
        return dict(kind=kind, dtype=rng.choice(["f32", "i32"]), batch=_log(rng, 1, 16),
                    M=_log(rng, 16, 2048), N=_log(rng, 16, 2048), K=_log(rng, 16, 1024),
                    ta=rng.randint(0, 1), tb=rng.randint(0, 1))
    return dict(kind=kind, L=rng.randint(6, 18))


# ---------------------------------------------------------------- inputs


def _rng(case, seed):
    return np.random.default_rng([int(seed)] + [ord(c) for c in case["kind"]])


def _signs(rng, shape):
    return np.where(rng.integers(0, 2, shape) == 0, -1.0, 1.0).astype(np.float32)


def _gauss(rng, shape, sigma=1.0):
    return (sigma * rng.standard_normal(shape)).astype(np.float32)


def _inputs(case, seed):
    """The host inputs of a case: graphs and couplings, from the seed alone."""
    rng = _rng(case, seed)
    k = case["kind"]
    if k == "single":
        inst = I.square_lattice(case["L"], seed=0)
        return dict(inst=inst, J=_signs(rng, len(inst["J"])))
    if k == "config":
        inst = I.square_lattice(case["L"], case["W"], coupling="gauss", field_sigma=0.1, seed=1)
        return dict(inst=inst, J=_gauss(rng, (case["B"], len(inst["J"]))),
                    h=_gauss(rng, (case["B"], inst["n"]), 0.1))
    if k == "mixed":
        # sides are part of the case, couplings of the seed
        sides = np.random.default_rng(2026).integers(case["Lmin"], case["Lmax"] + 1, case["B"])
        out = []
        for s in sides:
            inst = I.square_lattice(int(s), seed=0)
            out.append(dict(inst, J=_signs(rng, len(inst["J"]))))
        return dict(insts=out, sides=[int(s) for s in sides])
    if k == "chimera":
        inst = I.chimera(case["L"], seed=0)
        return dict(inst=inst, J=_signs(rng, len(inst["J"])))
    if k == "max2sat":
        sat = I.max2sat_regular3(case["N"], seed=case["graph"])
        sats = [dict(sat, clauses=np.where(rng.integers(0, 2, sat["clauses"].shape) == 1,
                                           -np.abs(sat["clauses"]),
                                           np.abs(sat["clauses"])).astype(np.int32))
                for _ in range(case["B"])]
        cp = [P.Max2SAT.couplings(x) for x in sats]
        return dict(sat=sats[0], J=np.stack([c[1] for c in cp]), h=np.stack([c[2] for c in cp]))
    if k == "rrg":
        inst = I.random_regular3(case["N"], seed=case["graph"])
        return dict(inst=inst, J=_gauss(rng, (case["B"], len(inst["J"]))))
    if k == "potts":
        inst = I.potts_square(case["L"], seed=0)
        return dict(inst=inst, J=_gauss(rng, (case["B"], len(inst["J"]))))
    if k == "cubic":
        inst = I.cubic_lattice(case["L"], case["W"], case["H"], coupling="gauss", seed=0)
        return dict(inst=inst, J=_gauss(rng, (case["B"], len(inst["J"]))))
    if k == "sample":
        inst = I.square_lattice(case["L"], seed=0)
        return dict(inst=dict(inst, J=_signs(rng, len(inst["J"]))), seed=int(rng.integers(1 << 30)))
    if k == "autograd":
        inst = I.square_lattice(case["L"], coupling="gauss", field_sigma=0.1, seed=1)
        return dict(inst=inst, J=_gauss(rng, len(inst["J"])), h=_gauss(rng, inst["n"], 0.1))
    raise ValueError(k)


def _gemm_inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    b, M, N, K = case["batch"], case["M"], case["N"], case["K"]
    sa = (b, K, M) if case["ta"] else (b, M, K)
    sb = (b, N, K) if case["tb"] else (b, K, N)
    if case["dtype"] == "f32":
        A = torch.randn(sa, generator=g, device="cuda") * 8
        Bm = torch.randn(sb, generator=g, device="cuda") * 8
    else:
        A = torch.randint(-40, 41, sa, generator=g, device="cuda", dtype=torch.int32)
        Bm = torch.randint(-40, 41, sb, generator=g, device="cuda", dtype=torch.int32)
    return A, Bm


def prepare(case, seed):
    k = case["kind"]
    if k == "gemm":
        A, Bm = _gemm_inputs(case, seed)
        C = torch.empty((case["batch"], case["M"], case["N"]), dtype=A.dtype, device="cuda")
        return dict(kind=k, A=A, B=Bm, C=C, ta=bool(case["ta"]), tb=bool(case["tb"]))
    d = _inputs(case, seed)
    dev = lambda a: torch.tensor(a, device="cuda")  # noqa: E731
    s = dict(kind=k)
    if k in ("single", "autograd"):
        s["sg"] = P.SpinGlass(d["inst"], order="sweep", seq=I.square_sweep_order(case["L"]))
        if k == "autograd":
            s.update(J=dev(d["J"]).requires_grad_(True), h=dev(d["h"]).requires_grad_(True))
        else:
            s["J"] = d["J"]
    elif k == "config":
        s.update(J=dev(d["J"]), h=dev(d["h"]),
                 sg=P.SpinGlass(d["inst"], order="greedy", seed=1, restarts=case["restarts"]))
    elif k == "mixed":
        s["sgs"] = [P.SpinGlass(x, order="sweep", seq=I.square_sweep_order(L))
                    for x, L in zip(d["insts"], d["sides"])]
        s["ctxs"] = [g.ctx for g in s["sgs"]]
    elif k == "chimera":
        s["J"] = d["J"]
        s["sg"] = P.SpinGlass(d["inst"], order="sweep", seq=I.chimera_sweep_order(case["L"]))
    elif k == "max2sat":
        s.update(J=d["J"], h=d["h"],
                 sg=P.Max2SAT(d["sat"], order="greedy", seed=1, restarts=128))
    elif k in ("rrg", "cubic"):
        s.update(J=dev(d["J"]), sg=P.SpinGlass(d["inst"], order="greedy", seed=1, restarts=128))
    elif k == "potts":
        s.update(J=dev(d["J"]), sg=P.SpinGlass(d["inst"], order="sweep",
                                               seq=I.square_sweep_order(case["L"])))
    elif k == "sample":
        s.update(seed=d["seed"], samples=case["samples"],
                 sg=P.SpinGlass(d["inst"], order="greedy", seed=1, restarts=64))
    return s


# ---------------------------------------------------------------- one pass


def _limbs(counts, per=4):
    """Counts (Python integers) as rows of little-endian 64-bit limbs."""
    mask = (1 << 64) - 1
    return np.array([[(int(c) >> (64 * j)) & mask for j in range(per)] for c in counts],
                    np.uint64).view(np.int64)


def run(state):
    k = state["kind"]
    if k == "gemm":
        B.tn_maxplus_gemm(state["A"], state["B"], state["C"], transA=state["ta"],
                          transB=state["tb"],
                          stream_handle=torch.cuda.current_stream().cuda_stream)
        return state["C"]
    if k == "mixed":
        st, E, counts, status = B.tn_batch_run(state["ctxs"], limbs_per=4)
        return {"E": E, "count": _limbs(counts), "status": status}
    sg = state["sg"]
    if k in ("single", "chimera"):
        # a new coupling set on a kept order: energy and degeneracy
        sg.set_couplings(state["J"])
        E = sg.energy()
        count, ln_count, E2 = sg.count(3)
        return {"E": E, "E_count": E2, "ln_count": ln_count, "count": _limbs([count])}
    if k == "max2sat":
        E, counts, status = sg.count_batch(state["J"], state["h"], 3, limbs_per=4)
        return {"E": E, "count": _limbs(counts), "status": status}
    if k == "sample":
        return sg.sample(state["samples"], seed=state["seed"])
    if k == "autograd":
        J, h = state["J"], state["h"]
        J.grad = h.grad = None
        E = P.TropicalEnergy.apply(J, h, sg)
        E.backward()
        return {"E": E.detach().float(), "dJ": J.grad, "dh": h.grad}
    E, sigma = sg.config_batch(state["J"], state.get("h"))
    return {"E": E.astype(np.float32), "sigma": sigma}


# ---------------------------------------------------------------- floors


def _frontier_work(n, w, q, updates_per_spin=1.0):
    """Tropical operations (an add and a max each) of moving a frontier of w spins
    over n spins, one spin at a time: q multiply-adds per state and spin."""
    return 2.0 * q * max(1, n - w) * float(q) ** w * updates_per_spin


def work(case):
    """What a pass cannot do without: the couplings in and the results out, and the
    max-plus operations of sweeping the narrowest frontier of the graph (a counting
    tuple costs two operations more per multiply-add)."""
    k = case["kind"]
    if k == "gemm":
        b, M, N, K = case["batch"], case["M"], case["N"], case["K"]
        return dict(bytes=4.0 * b * (M * K + K * N + M * N), flops=2.0 * b * M * N * K)
    if k == "mixed":
        sides = np.random.default_rng(2026).integers(case["Lmin"], case["Lmax"] + 1, case["B"])
        return dict(bytes=float(sum(4 * 2 * s * (s - 1) + 40 for s in sides)),
                    flops=float(sum(2 * _frontier_work(int(s) ** 2, int(s), 2) for s in sides)))
    if k in ("single", "autograd", "sample", "potts"):
        n, w, m = case["L"] ** 2, case["L"], 2 * case["L"] * (case["L"] - 1)
    elif k == "config":
        n, w = case["L"] * case["W"], min(case["L"], case["W"])
        m = 2 * n
    elif k == "chimera":
        n, w, m = 8 * case["L"] ** 2, 4 * case["L"], 24 * case["L"] ** 2
    elif k == "cubic":
        n = case["L"] * case["W"] * case["H"]
        w, m = n // max(case["L"], case["W"], case["H"]), 3 * n
    else:   # random 3-regular graphs: treewidth about N / 8
        n, w, m = case["N"], case["N"] // 8, 3 * case["N"] // 2
    q = 3 if k == "potts" else 2
    # greedy orders grow the frontier from several sides and hold its full width
    # for part of the spins only (measured on the 24 x 24 and 5 x 5 x 5 orders)
    part = {"config": 0.35, "cubic": 0.08}.get(k, 1.0)
    per = _frontier_work(n, w, q, part)
    if k == "single" or k == "chimera":
        per *= 3          # the energy, then the counting tuples
    elif k == "max2sat":
        per *= 2
    elif k == "sample":
        per *= 2 * 2 * n  # two candidates per spin and sample
    reps = case.get("B", 1) * case.get("samples", 1)
    return dict(bytes=float(reps * (4 * (m + n) + n + 8)), flops=per * reps)


# ---------------------------------------------------------------- 64-bit results


def _frontier(n, q, w, mats, diag):
    """max over all states of the sum of pair terms, and one maximising state.

    mats[i]: {j: (q, q) array, indexed [s_j, s_i]} for the earlier neighbours j >= i - w
    of spin i; diag[i]: (q,) array.  One pass over the spins with a frontier of the
    last w of them (spin j on leg j mod w), in float64.
    """
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    T = torch.full((q ** w,), -float("inf"), dtype=torch.float64, device=dev)
    T[0] = 0.0
    back = []
    for i in range(n):
        p = i % w
        hi, lo = q ** p, q ** (w - 1 - p)
        M = torch.zeros((q, q), dtype=torch.float64)
        if i - w in mats[i]:
            M = M + torch.as_tensor(mats[i][i - w])
        M = (M + torch.as_tensor(diag[i])[None, :]).to(dev)
        V = T.view(hi, q, lo)
        out = torch.empty_like(V)
        arg = torch.empty(V.shape, dtype=torch.uint8, device=dev)
        for s in range(q):
            best, at = V[:, 0] + M[0, s], torch.zeros_like(arg[:, 0])
            for o in range(1, q):
                c = V[:, o] + M[o, s]
                at = torch.where(c > best, torch.full_like(at, o), at)
                best = torch.maximum(best, c)
            out[:, s], arg[:, s] = best, at
        back.append(arg.view(-1))
        T = out.view(-1)
        for j, Mj in mats[i].items():
            if j == i - w:
                continue
            a, b = sorted((p, j % w))
            Mt = torch.as_tensor(Mj).to(dev)
            if a == p:
                Mt = Mt.t()
            T = (T.view(q ** a, q, q ** (b - a - 1), q, -1) + Mt[None, :, None, :, None]).view(-1)
    top = int(torch.argmax(T))
    best = float(T[top])
    digits = [(top // q ** (w - 1 - p)) % q for p in range(w)]
    state = np.zeros(n, np.int64)
    for i in range(n - 1, -1, -1):
        p = i % w
        state[i] = digits[p]
        at = sum(d * q ** (w - 1 - j) for j, d in enumerate(digits))
        digits[p] = int(back[i][at])
    return best, state


def _ising_exact(inst, J, h, w):
    mats = [dict() for _ in range(inst["n"])]
    s = np.array([1.0, -1.0])
    for (u, v), j in zip(np.asarray(inst["edges"]), J):
        u, v = int(min(u, v)), int(max(u, v))
        mats[v][u] = float(j) * np.outer(s, s)
    z = np.zeros(2)
    diag = [z if h is None else float(h[i]) * s for i in range(inst["n"])]
    best, state = _frontier(inst["n"], 2, w, mats, diag)
    return -best, 1 - 2 * state


def exact(case, seed):
    k = case["kind"]
    if k == "gemm":
        A, Bm = _gemm_inputs(case, seed)
        if case["dtype"] != "f32":
            return None
        A = (A.transpose(1, 2) if case["ta"] else A).double().contiguous()
        Bm = (Bm.transpose(1, 2) if case["tb"] else Bm).double().contiguous()
        C = torch.full((A.shape[0], A.shape[1], Bm.shape[2]), -float("inf"), dtype=torch.float64,
                       device=A.device)
        for x in range(A.shape[2]):
            torch.maximum(C, A[:, :, x:x + 1] + Bm[:, x:x + 1, :], out=C)
        return C
    if k == "config":
        d = _inputs(case, seed)
        L, W = case["L"], case["W"]
        inst = d["inst"]
        if W > L:   # number the spins along the longer side
            e = np.asarray(inst["edges"])
            inst = dict(inst, edges=(e % W) * L + e // W)
            perm = (np.arange(L * W) % W) * L + np.arange(L * W) // W
        else:
            perm = np.arange(L * W)
        E, S = [], []
        for b in range(case["B"]):
            h = np.empty(L * W, np.float32)
            h[perm] = d["h"][b]
            e, s = _ising_exact(inst, d["J"][b], h, min(L, W))
            E.append(e)
            S.append(s[perm])
        return {"E": np.array(E), "sigma": np.array(S, np.int8)}
    if k == "autograd":
        d = _inputs(case, seed)
        E, s = _ising_exact(d["inst"], d["J"], d["h"], case["L"])
        e = np.asarray(d["inst"]["edges"])
        return {"E": torch.tensor(E, dtype=torch.float64),
                "dJ": torch.tensor(-(s[e[:, 0]] * s[e[:, 1]]).astype(np.float64)),
                "dh": torch.tensor(-s.astype(np.float64))}
    if k == "potts":
        d = _inputs(case, seed)
        E = []
        for b in range(case["B"]):
            mats = [dict() for _ in range(d["inst"]["n"])]
            for (u, v), j in zip(np.asarray(d["inst"]["edges"]), d["J"][b]):
                mats[int(max(u, v))][int(min(u, v))] = float(j) * np.eye(3)
            best, _ = _frontier(d["inst"]["n"], 3, case["L"], mats,
                                [np.zeros(3)] * d["inst"]["n"])
            E.append(-best)
        return {"E": np.array(E), "sigma": None}
    if k == "cubic":
        d = _inputs(case, seed)
        L, W, H = case["L"], case["W"], case["H"]
        # number the spins layer by layer along the longest side
        axes = sorted(range(3), key=lambda a: -(L, W, H)[a])
        ids = np.arange(L * W * H).reshape(L, W, H).transpose(axes).reshape(-1)
        at = np.empty_like(ids)
        at[ids] = np.arange(len(ids))
        inst = dict(d["inst"], edges=at[np.asarray(d["inst"]["edges"])])
        w = L * W * H // max(L, W, H)
        return {"E": np.array([_ising_exact(inst, d["J"][b], None, w)[0]
                               for b in range(case["B"])]), "sigma": None}
    return None
