"""What a user of this framework has it compute, as cases that can be timed and checked.

Three layouts, as in the repository's own workloads: boxes on a line or a
lattice (the tiny chain, the alkane chain, the lattices of 40^3 boxes) and
uneven boxes along a random walk (the amorphous polymer).  Four kinds of work:

  assemble  the H / S blocks from resident states (optionally after a new
            potential), read into a device array
  eigs      the fragment eigenstates of every box
  window    the assembly followed by Eq. 2 in an energy window
  pencil    products of the assembled pencil with a block of vectors
"""
import collections
import itertools
import math
import random

import numpy as np
import torch

from paper_1011_4764_gb300 import ofm

Grid = collections.namedtuple("Grid", "n h")
Box = collections.namedtuple("Box", "off ext n_states")
SPACING = 0.5   # bohr, as in every workload of the repository


def _case(name, kind, layout, count, box, stride, states, precision, storage="fp32", **more):
    c = {"name": name, "kind": kind, "layout": layout, "states": states, "precision": precision,
         "storage": storage, "open": False, "new_potential": False, "vectors": False, "columns": 0}
    for d, k in enumerate("xyz"):
        c["count_" + k], c["box_" + k], c["stride_" + k] = count[d], box[d], stride[d]
    c.update(more)
    return c


def listed():
    return [
        # the tiny chain in FP64, assembly and window: the smallest calls, all launches and latency
        _case("step_tiny_fp64", "window", "lattice", (4, 1, 1), (16, 12, 12), (8, 12, 12), 6, "fp64", "fp64"),
        # the alkane chain's assembly in the default mixed arithmetic: an ordinary small system
        _case("asm_alkane_bf16x3", "assemble", "lattice", (31, 1, 1), (16, 32, 32), (8, 32, 32), 32, "bf16x3", open=True),
        # 4x4x4 cells of the large lattice: an ordinary three-dimensional system
        _case("asm_lattice_bf16x3", "assemble", "lattice", (4, 4, 4), (40, 40, 40), (24, 24, 24), 96, "bf16x3"),
        # 8x8x4 cells after a new potential, the step of an outer loop over potentials: the largest
        # (the same kernels as the 16x8x8 lattice at a quarter of its size)
        _case("asm_large_bf16x3", "assemble", "lattice", (8, 8, 4), (40, 40, 40), (24, 24, 24), 96, "bf16x3", new_potential=True),
        # uneven boxes with uneven state counts, in TF32: the polymer's assembly
        _case("asm_polymer_tf32", "assemble", "ragged", (56, 1, 1), (16, 16, 16), (40, 40, 40), 64, "tf32"),
        # plain FP32 arithmetic, what the mixed precisions are checked against; odd sizes and states
        _case("asm_lattice_fp32", "assemble", "lattice", (3, 3, 3), (31, 29, 27), (19, 17, 17), 45, "fp32"),
        # fragment states of the alkane chain
        _case("eigs_alkane_fp32", "eigs", "lattice", (31, 1, 1), (16, 32, 32), (8, 32, 32), 32, "fp32", open=True),
        # fragment states of the lattice: the longest step of a calculation on the largest systems
        _case("eigs_lattice_fp32", "eigs", "lattice", (3, 3, 3), (40, 40, 40), (24, 24, 24), 96, "fp32"),
        # fragment states of a few uneven boxes in FP64 (parity runs)
        _case("eigs_ragged_fp64", "eigs", "ragged", (12, 1, 1), (12, 12, 12), (24, 24, 24), 24, "fp64", "fp64"),
        # the alkane chain's assembly and every level within 0.3 Ha above an index (n = 992)
        _case("window_alkane", "window", "lattice", (31, 1, 1), (16, 32, 32), (8, 32, 32), 32, "bf16x3", open=True),
        # the lowest levels with their coefficient vectors, FP64 throughout, an odd-sized chain
        _case("window_vectors_fp64", "window", "lattice", (15, 1, 1), (16, 21, 19), (9, 21, 19), 21, "fp64", "fp64", open=True, vectors=True),
        # H X and S X for a block of vectors, as an iterative solver of Eq. 2 asks for
        _case("pencil_lattice", "pencil", "lattice", (4, 4, 4), (20, 20, 20), (12, 12, 12), 96, "fp64", columns=16),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case of these ranges, at most as costly as the largest listed ones."""
    kind = rng.choice(["assemble", "assemble", "assemble", "eigs", "eigs", "window", "pencil"])
    if kind == "window":   # chains, from the tiny one to about the alkane chain's basis
        vectors = rng.random() < 0.4
        n = _log_int(rng, 4, 31)
        y, z = rng.randint(12, 32), rng.randint(12, 32)
        states = min(rng.randint(5, 32), 600 // n if vectors else 992 // n)
        fp64 = vectors or rng.random() < 0.3
        return _unnamed(kind, "lattice", (n, 1, 1), (16, y, z), (rng.choice([8, 9, 10]), y, z), max(4, states),
                        "fp64" if fp64 else "bf16x3", "fp64" if fp64 else "fp32", open=True, vectors=vectors)
    if kind == "pencil":
        e = rng.randint(12, 20)
        s = int(round(0.6 * e))
        return _unnamed(kind, "lattice", tuple(rng.randint(2, 4) for _ in range(3)), (e, e, e), (s, s, s),
                        rng.randint(8, 96), "fp64", columns=_log_int(rng, 1, 64))
    layout = rng.choice(["chain", "lattice", "ragged"])
    if kind == "eigs":
        storage = rng.choice(["fp32", "fp32", "fp64"])
        top = 2.0e7 if storage == "fp32" else 1.0e6   # points x states over all boxes
        precision = storage
    else:
        storage = "fp32"
        precision = rng.choice(["bf16x3", "bf16x3", "bf16", "tf32", "fp32", "fp64"])
        top = {"fp64": 8.0e6, "fp32": 1.2e8}.get(precision, 1.2e9)
    if layout == "ragged":
        lo = rng.choice([12, 16])
        hi = lo + 8 * rng.randint(1, 2 if kind == "eigs" else 3)
        states = rng.randint(9, 24 if kind == "eigs" else 64)
        n = _log_int(rng, 6, 12 if kind == "eigs" else 60)
        while n > 2 and n * ((lo + hi) / 2.0) ** 3 * states > top:
            n -= 1
        return _unnamed(kind, layout, (n, 1, 1), (lo,) * 3, (hi,) * 3, states, precision, storage,
                        shape=rng.randint(0, 999))
    if layout == "chain":
        y, z = rng.choice([12, 20, 27, 32]), rng.choice([12, 19, 32])
        box, stride = (16, y, z), (rng.choice([8, 9]), y, z)
        states = rng.randint(6, 32)
        most = (_log_int(rng, 4, 64), 1, 1)
    else:
        small = kind == "eigs" and storage == "fp64"
        e = [rng.randint(14, 22) if small else rng.randint(18, 40) for _ in range(3)]
        box, stride = tuple(e), tuple(int(round(0.6 * v)) for v in e)
        states = rng.randint(6, 24) if small else rng.randint(12, 96)
        most = tuple(_log_int(rng, 2, 8) for _ in range(3))
    count = list(most)
    while math.prod(count) * math.prod(box) * states > top and max(count) > 2:
        count[count.index(max(count))] -= 1
    return _unnamed(kind, "lattice", tuple(count), box, stride, states, precision, storage,
                    open=layout == "chain", new_potential=kind == "assemble" and rng.random() < 0.3)


def _unnamed(*a, **k):
    c = _case("", *a, **k)
    del c["name"]
    return c


def _geometry(case):
    """The grid and the boxes: of the case alone, whatever the seed."""
    count, box, stride = ([case[w + k] for k in "xyz"] for w in ("count_", "box_", "stride_"))
    if case["layout"] == "lattice":
        n = [c * s if c > 1 else b for c, s, b in zip(count, stride, box)]
        if case["open"] and count[0] > 1:
            n[0] = (count[0] - 1) * stride[0] + box[0]
        ext = [b if b != m - 1 else b - 1 for b, m in zip((min(b, m) for b, m in zip(box, n)), n)]
        boxes = [Box((i * stride[0], j * stride[1], k * stride[2]), tuple(ext), case["states"])
                 for k in range(count[2]) for j in range(count[1]) for i in range(count[0])]
        return Grid(tuple(n), SPACING), boxes
    # uneven boxes along a random walk; edges are multiples of 4 from box_* to stride_*
    lo, hi = case["box_x"], case["stride_x"]
    r = random.Random(1000 + case.get("shape", 0))
    n = max(hi + 8, 8 * int(math.ceil(hi * (count[0] / 3.0) ** (1.0 / 3.0) / 8.0)))
    at, boxes = [r.uniform(0, n) for _ in range(3)], []
    for _ in range(count[0]):
        ext = tuple(r.randrange(lo, hi + 1, 4) for _ in range(3))
        states = r.randint(max(1, case["states"] // 8), case["states"])
        boxes.append(Box(tuple(int(round(a - 0.5 * e)) % n for a, e in zip(at, ext)), ext, states))
        step = [r.gauss(0, 1) for _ in range(3)]
        s = 0.45 * (lo + hi) / 2 / math.sqrt(sum(v * v for v in step))
        at = [a + s * v for a, v in zip(at, step)]
    return Grid((n, n, n), SPACING), boxes


def _potential(grid, gen):
    """Gaussian wells (depth 0.6 to 1.2 Ha, width 0.8 bohr) at random grid points, about
    as dense as in the repository's lattices: float64, [z][y][x]."""
    nx, ny, nz = grid.n
    npts = nx * ny * nz
    wells = max(4, int(1.4e-3 * npts))
    V = torch.zeros(npts, dtype=torch.float64, device="cuda")
    where = torch.randperm(npts, generator=gen, device="cuda")[:wells]
    V[where] = -(0.6 + 0.6 * torch.rand(wells, generator=gen, device="cuda", dtype=torch.float64))
    k2 = 0
    for d, n in enumerate((nz, ny, nx)):
        k = 2.0 * math.pi * torch.fft.fftfreq(n, grid.h, dtype=torch.float64, device="cuda")
        shape = [1, 1, 1]
        shape[d] = n
        k2 = k2 + (k * k).reshape(shape)
    w = 0.8
    weight = (2.0 * math.pi) ** 1.5 * (w / grid.h) ** 3
    V = torch.fft.ifftn(torch.fft.fftn(V.reshape(nz, ny, nx)) * torch.exp(-0.5 * w * w * k2)).real
    return (weight * V).contiguous()


def _modes(ext, count):
    """The `count` lowest particle-in-a-box modes of a box, orthonormal: (count, points) float32."""
    top = [min(e, 24) for e in ext]
    k = sorted(itertools.product(*(range(1, t + 1) for t in top)),
               key=lambda q: (sum((v / (e + 1.0)) ** 2 for v, e in zip(q, ext)), q))[:count]
    one = []
    for d, e in enumerate(ext):
        i = torch.arange(1, e + 1, dtype=torch.float64, device="cuda")
        q = torch.tensor([v[d] for v in k], dtype=torch.float64, device="cuda")
        one.append((math.sqrt(2.0 / (e + 1)) * torch.sin(math.pi / (e + 1) * q[:, None] * i[None])).float())
    x, y, z = one
    return (z[:, :, None, None] * y[:, None, :, None] * x[:, None, None, :]).reshape(len(k), -1)


def _states(boxes, gen):
    """Smooth orthonormal states of every box, lowest modes first: yields (n_states, points)
    float64 tensors whose values are FP32 numbers (the storage precision)."""
    known = {}
    for b in boxes:
        points = math.prod(b.ext)
        key = (b.ext, b.n_states)
        if key not in known:
            z = _modes(b.ext, min(points, 2 * b.n_states))
            mix = torch.exp(-4.0 * torch.abs(torch.arange(len(z), device="cuda")[:, None]
                                             - torch.arange(b.n_states, device="cuda")[None]) / b.n_states)
            if len(known) > 8:
                known.clear()
            known[key] = (z, mix)
        z, mix = known[key]
        c = torch.randn(mix.shape, generator=gen, device="cuda") * mix
        c[:b.n_states] += 3.0 * torch.eye(b.n_states, device="cuda")
        q, _ = torch.linalg.qr(c)
        yield (q.T @ z).double().contiguous()


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


class _State:
    pass


def prepare(case, seed):
    gen = _generator(seed)
    s = _State()
    s.case = case
    s.stream = torch.cuda.Stream()
    with torch.cuda.stream(s.stream):
        grid, boxes = _geometry(case)
        V = _potential(grid, gen)
        s.ctx = ofm.Context(s.stream)
        s.ctx.build_fragments(grid, V, boxes, storage=case["storage"])
        s.basis = sum(b.n_states for b in boxes)
        if case["kind"] != "eigs":
            for a, phi in enumerate(_states(boxes, gen)):
                s.ctx.set_fragment_states(a, phi)
        if case["kind"] == "assemble":
            s.V = _potential(grid, gen) if case["new_potential"] else None
            s.ctx.assemble(case["precision"])
            s.out = torch.zeros(s.ctx.blocks_count(), dtype=torch.float64, device="cuda")
        elif case["kind"] == "window" and case["vectors"]:
            # an energy window that holds the lowest levels
            s.levels = max(1, s.basis // 10)
            s.ctx.assemble(case["precision"])
            E = s.ctx.eigs_by_index(0, s.levels + 1)
            s.window = (float(E[0]) - 0.05, 0.5 * float(E[-2] + E[-1]))
        elif case["kind"] == "window":
            s.first = s.basis // 5
        elif case["kind"] == "pencil":
            s.ctx.assemble(case["precision"])
            s.X = torch.randn((case["columns"], s.basis), generator=gen, dtype=torch.float64, device="cuda")
            s.Y = [torch.zeros_like(s.X) for _ in range(2)]
        s.stream.synchronize()
    return s


def run(s):
    case, ctx = s.case, s.ctx
    with torch.cuda.stream(s.stream):
        if case["kind"] == "eigs":
            eps, _, _ = ctx.fragment_eigs(allow_not_converged=True)
            # energies of FP32 states are FP32 numbers; their residuals are below the tolerance
            return eps.astype(np.float32) if case["storage"] == "fp32" else eps
        if case["kind"] == "pencil":
            return [ctx.pencil_apply(w, s.X, out=y) for w, y in zip("HS", s.Y)]
        if case["kind"] == "assemble":
            if s.V is not None:
                ctx.set_potential(s.V)
            ctx.assemble(case["precision"])
            ctx.get_blocks(out=s.out)
            # blocks of the mixed and FP32 arithmetics are kept as FP32
            return s.out if case["precision"] == "fp64" else s.out.float()
        ctx.assemble(case["precision"])
        if case["vectors"]:
            E, C, _ = ctx.window_eigs(*s.window, max_out=s.levels, vectors=True)
            return [E, _gauge(C)]
        E, count = ctx.window_from_index(s.first, 0.3)
        levels = np.zeros(s.basis, dtype=np.float64 if case["precision"] == "fp64" else np.float32)
        levels[:count] = E
        return [levels, count]


def _gauge(C):
    """Each column with its largest component positive."""
    top = np.abs(C).argmax(axis=0)
    return C * np.sign(C[top, np.arange(C.shape[1])])[None]


def _pairs(grid, boxes):
    """Pairs a <= b whose boxes meet (b's grown by one point), with the shared points of
    B_a and B_b+ per dimension as index pairs (in a's box, in b's grown box)."""
    nd = [grid.n[d] for d in range(3)]

    def meet(a, b, d):
        n = nd[d]
        grown = b.ext[d] < n
        first = (b.off[d] - (1 if grown else 0)) % n
        length = b.ext[d] + (2 if grown else 0)
        i = np.arange(a.ext[d])
        j = (a.off[d] + i - first) % n
        keep = j < length
        return i[keep], j[keep]

    known, out = {}, []
    for i, a in enumerate(boxes):
        for k in range(i, len(boxes)):
            b, shared = boxes[k], []
            for d in range(3):
                key = (d, a.ext[d], b.ext[d], (a.off[d] - b.off[d]) % nd[d])
                if key not in known:
                    known[key] = meet(a, b, d)
                shared.append(known[key])
                if not len(shared[-1][0]):
                    break
            else:
                out.append((i, k, shared))
    return out


def _counts(case):
    grid, boxes = _geometry(case)
    flops = values = 0
    for a, b, shared in _pairs(grid, boxes):
        points = math.prod(len(i) for i, _ in shared)
        inner = 1   # |B_a n B_b|: the points of B_b itself
        for d, (_, j) in enumerate(shared):
            e, n = boxes[b].ext[d], grid.n[d]
            inner *= int(np.sum((j >= 1) & (j <= e))) if e < n else len(j)
        flops += 2 * boxes[a].n_states * boxes[b].n_states * (points + inner)
        values += 2 * boxes[a].n_states * boxes[b].n_states
    return grid, boxes, flops, values


def work(case):
    es = 8 if case["storage"] == "fp64" else 4
    grid, boxes, flops, values = _counts(case)
    points = math.prod(grid.n)
    states = sum(math.prod(b.ext) * b.n_states for b in boxes)
    n = sum(b.n_states for b in boxes)
    if case["kind"] == "eigs":   # V in, states out; one H apply and one Rayleigh-Ritz of the block
        return {"bytes": es * (points + states),
                "flops": sum(math.prod(b.ext) * b.n_states * (10 + 4 * b.n_states) for b in boxes)}
    if case["kind"] == "pencil":   # blocks and X once, both products
        return {"bytes": 8 * (values + 3 * n * case["columns"]), "flops": 4 * values * case["columns"]}
    total = {"bytes": es * (points + states) + 8 * values, "flops": flops + 10 * states}
    if case["kind"] == "window":   # Cholesky, two triangular reductions, tridiagonalisation
        total["flops"] += int(n ** 3 * (1 / 3 + 1 + 4 / 3))
    return total


# ---------------------------------------------------------------- in 64 bits

def _grow(phi, box, grid):
    """(n, points) on the box -> (n, z, y, x) on the grown box, zero halo."""
    x, y, z = box.ext
    pad = []
    for d in range(3):
        pad += [1, 1] if box.ext[d] < grid.n[d] else [0, 0]
    return torch.nn.functional.pad(phi.reshape(-1, z, y, x), pad)


def _neighbours(f, wrap):
    """Sum of the six neighbours of (n, z, y, x); wrap[d] for d = x, y, z."""
    total = torch.zeros_like(f)
    for d in range(3):
        axis = 3 - d
        for s in (1, -1):
            g = torch.roll(f, s, axis)
            if not wrap[d]:
                edge = [slice(None)] * 4
                edge[axis] = 0 if s == 1 else -1
                g[tuple(edge)] = 0
            total += g
    return total


def _local_potential(V, box, grid, grown):
    idx = []
    for d in range(3):
        g = 1 if grown and box.ext[d] < grid.n[d] else 0
        idx.append((torch.arange(box.ext[d] + 2 * g, device="cuda") + box.off[d] - g) % grid.n[d])
    return V[idx[2]][:, idx[1]][:, :, idx[0]]


def _blocks(grid, boxes, V, states):
    """Every [H_ab, S_ab] in 64 bits."""
    full = [tuple(b.ext[d] == grid.n[d] for d in range(3)) for b in boxes]
    phis, hphis = [], []
    for b, w, phi in zip(boxes, full, states):
        f = _grow(phi, b, grid)
        v = _local_potential(V, b, grid, True)
        phis.append(f)
        hphis.append((3.0 / grid.h ** 2 + v) * f - 0.5 / grid.h ** 2 * _neighbours(f, w))
    out = []
    for a, b, shared in _pairs(grid, boxes):
        ia = [torch.as_tensor(i, device="cuda") + (0 if full[a][d] else 1) for d, (i, _) in enumerate(shared)]
        ib = [torch.as_tensor(j, device="cuda") for _, j in shared]

        def at(f, i):
            return f[:, i[2][:, None, None], i[1][None, :, None], i[0][None, None, :]].reshape(f.shape[0], -1)
        A = at(phis[a], ia)
        H, S = A @ at(hphis[b], ib).T, A @ at(phis[b], ib).T
        if a == b:
            H, S = 0.5 * (H + H.T), 0.5 * (S + S.T)
        out.append((a, b, H, S))
    return out


def _dense(boxes, blocks):
    at = np.concatenate([[0], np.cumsum([b.n_states for b in boxes])])
    H = torch.zeros((int(at[-1]),) * 2, dtype=torch.float64, device="cuda")
    S = torch.zeros_like(H)
    for a, b, h, s in blocks:
        H[at[a]:at[a + 1], at[b]:at[b + 1]] = h
        H[at[b]:at[b + 1], at[a]:at[a + 1]] = h.T
        S[at[a]:at[a + 1], at[b]:at[b + 1]] = s
        S[at[b]:at[b + 1], at[a]:at[a + 1]] = s.T
    return H, S


def _levels(H, S):
    L = torch.linalg.cholesky(S)
    A = torch.linalg.solve_triangular(L, H, upper=False)
    A = torch.linalg.solve_triangular(L, A.T, upper=False)
    E, X = torch.linalg.eigh(0.5 * (A + A.T))
    return E, torch.linalg.solve_triangular(L.T, X, upper=True)


def _lowest(grid, box, V, n):
    """The n lowest eigenvalues of one box's H (zero outside the box, periodic where the box
    spans the grid), by a filtered subspace iteration in 64 bits; None if it did not settle."""
    points = math.prod(box.ext)
    x, y, z = box.ext
    v = _local_potential(V, box, grid, False)
    wrap = tuple(box.ext[d] == grid.n[d] for d in range(3))

    def apply(f):
        f = f.reshape(-1, z, y, x)
        return ((3.0 / grid.h ** 2 + v) * f - 0.5 / grid.h ** 2 * _neighbours(f, wrap)).reshape(f.shape[0], -1)
    if points <= 3000:
        return torch.linalg.eigvalsh(apply(torch.eye(points, dtype=torch.float64, device="cuda")))[:n]
    m = min(points, n + max(8, n // 2))
    X = torch.randn((m, points), generator=_generator(1), dtype=torch.float64, device="cuda")
    top = 6.0 / grid.h ** 2 + float(V.max())
    low, cut, degree = None, None, 30
    for it in range(60):
        if cut is not None:
            e, c = 0.5 * (top - cut), 0.5 * (top + cut)
            s1 = e / (low - c)
            s, P, X = s1, X, (apply(X) - c * X) * (s1 / e)
            for _ in range(degree - 1):
                t = 1.0 / (2.0 / s1 - s)
                P, X, s = X, (apply(X) - c * X) * (2.0 * t / e) - s * t * P, t
        X = torch.linalg.qr(X.T)[0].T.contiguous()
        HX = apply(X)
        theta, Q = torch.linalg.eigh(X @ HX.T)
        X, HX = Q.T @ X, Q.T @ HX
        low, cut = float(theta[0]), float(theta[-1])
        if float((HX[:n] - theta[:n, None] * X[:n]).norm(dim=1).max()) < 1e-7:
            return theta[:n]   # the energies are exact to the square of that
    return None


def exact(case, seed):
    gen = _generator(seed)
    grid, boxes = _geometry(case)
    V = _potential(grid, gen)
    if case["kind"] == "eigs":
        if sum(math.prod(b.ext) * b.n_states for b in boxes) > 6.0e7:
            return None   # longer than is worth waiting for
        found = [_lowest(grid, b, V, b.n_states) for b in boxes]
        return None if any(f is None for f in found) else torch.cat(found)
    states = list(_states(boxes, gen))
    if case["kind"] == "assemble" and case["new_potential"]:
        V = _potential(grid, gen)
    blocks = _blocks(grid, boxes, V, states)
    if case["kind"] == "assemble":
        return torch.cat([m.reshape(-1) for _, _, H, S in blocks for m in (H, S)])
    H, S = _dense(boxes, blocks)
    n = H.shape[0]
    if case["kind"] == "pencil":
        X = torch.randn((case["columns"], n), generator=gen, dtype=torch.float64, device="cuda")
        return [X @ H, X @ S]
    E, C = _levels(H, S)
    if case["vectors"]:
        k = max(1, n // 10)
        return [E[:k].cpu().numpy(), _gauge(C[:, :k].cpu().numpy())]
    first = n // 5
    inside = E[first:][E[first:] <= E[first] + 0.3]
    levels = torch.zeros(n, dtype=torch.float64, device="cuda")
    levels[:len(inside)] = inside
    return [levels, None]
