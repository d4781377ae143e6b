"""Workloads of the block-forest DG library, as a user's program calls it.

Every case is one call sequence through the binding: a state is handed over
(``set_state``), marched by a number of SSP-RK3 time increments (``rk_step``,
or ``Batch.step`` for several forests together) and read back
(``get_state``).  The forests are lattices of root blocks of the unit cube (or
of [0,10]^2), with the shapes, degrees, precisions and options of the
repository's benchmark, adaptive and serving runs.

``exact`` advances the same input in FP64 with plain torch: nodal DG on the
Gauss points of an axis-aligned multi-level lattice of trilinear cells, all
blocks in one global frame (blocks of rotated roots are permuted into it and
back), guard traces by the split and the J-weighted combine.
"""
import itertools
import math

import numpy as np
import torch

import paper_2502_12620_gb300 as dgf

GAMMA = 1.4
PRECISION = {"fp32": dgf.FP32, "fp64": dgf.FP64, "fp32_comp": dgf.FP32_COMP}


# ------------------------------------------------------------------- cases
def _case(**kw):
    c = dict(kind="march", dim=3, B=2, extent=1.0, n_seg=8, p=2, precision="fp32", jitter=0.0, rotate=False,
             refine="none", initial="vortex", nonconforming="paper", limiter=0.0, cfl=0.1, steps=10)
    c.update(kw)
    return c


def listed():
    jitter3d = dict(B=2, jitter=0.1, rotate=True, refine="twice_centre")
    return [
        # the 2D isentropic-vortex run: the smallest forest, every launch counts
        _case(name="vortex2d_fp64_28leaves", dim=2, B=4, extent=10.0, precision="fp64", refine="centre", steps=20),
        # the benchmark's forest: jittered rotated roots with level jumps
        _case(name="jitter3d_p2_fp32_71leaves", steps=20, **jitter3d),
        # the same forest in the reference precision
        _case(name="jitter3d_p2_fp64_71leaves", precision="fp64", steps=4, **jitter3d),
        # the same forest with the state accumulated in FP64
        _case(name="jitter3d_p2_comp_71leaves", precision="fp32_comp", steps=10, **jitter3d),
        # the same forest with the conservative level-jump option
        _case(name="jitter3d_p2_mortar_71leaves", nonconforming="mortar", steps=10, **jitter3d),
        # the smallest solve of the serving mix
        _case(name="cube4_p1_fp32_64leaves", B=4, p=1, steps=20),
        # states above the L2 cache: single-level cubes of 16^3 roots
        _case(name="cube16_p1_fp32_4096leaves", B=16, p=1, initial="smooth", steps=4),
        _case(name="cube16_p2_fp32_4096leaves", B=16, p=2, initial="smooth", steps=4),
        # the highest degree, a mid-sized solve of the serving mix
        _case(name="cube8_p3_fp32_512leaves", B=8, p=3, steps=4),
        # adaptive blast between regrids: three levels, positivity limiter on
        _case(name="blast_amr_p1_limited", B=4, p=1, refine="shell", initial="blast", limiter=1e-6, steps=10),
        # adaptive cycle: march, indicator, refine, march, coarsen again
        _case(name="regrid_cycle_p1", kind="cycle", B=4, p=1, refine="shell2", initial="blast", limiter=1e-6, steps=10),
        # one round of the batched server: members admitted, marched together
        _case(name="batch_p2_5_8_10roots", kind="batch", members="5,8,10", B=10, p=2, initial="smooth", steps=8),
    ]


def draw(rng):
    """A case of the listed ones' ranges (sizes log-uniform, odd counts among them)."""
    log = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))  # noqa: E731
    family = rng.choice(["2d", "curved", "cube", "cube", "amr", "batch", "cycle"])
    p, cfl = rng.choice([1, 2, 3]), round(rng.uniform(0.03, 0.06), 4)
    if family == "2d":
        return _case(dim=2, B=log(3, 12), extent=10.0, n_seg=rng.choice([4, 8]), p=p, precision=rng.choice(["fp64", "fp32"]),
                     refine=rng.choice(["none", "centre"]), initial=rng.choice(["vortex", "smooth"]), cfl=cfl,
                     steps=rng.randint(3, 20))
    if family == "curved":
        precision = rng.choice(["fp32", "fp32", "fp64", "fp32_comp"])
        fp64 = precision == "fp64"  # the slowest precision: the smaller sizes
        return _case(B=2 if fp64 else rng.choice([2, 2, 3]), n_seg=rng.choice([4, 8, 8]), p=min(p, 2) if fp64 else p,
                     jitter=rng.uniform(0.02, 0.1), rotate=rng.choice([True, True, False]),
                     refine=rng.choice(["none", "twice_centre"]), precision=precision,
                     nonconforming=rng.choice(["paper", "paper", "mortar"]),
                     initial=rng.choice(["vortex", "smooth"]), cfl=cfl, steps=rng.randint(2, 4 if fp64 else 8))
    if family == "cube":
        return _case(B=log(3, {1: 16, 2: 14, 3: 8}[p]), p=p, initial=rng.choice(["vortex", "smooth"]),
                     cfl=cfl, steps=rng.randint(2, 5))
    if family == "amr":
        p = rng.choice([1, 2])
        return _case(B=rng.choice([3, 4, 5]), p=p, refine=rng.choice(["shell", "shell2"]), initial="blast",
                     limiter=rng.choice([0.0, 1e-6]) if p == 1 else 0.0, cfl=cfl, steps=rng.randint(2, 10))
    if family == "cycle":
        return _case(kind="cycle", B=rng.choice([3, 4, 5]), p=rng.choice([1, 2]), refine="shell2", initial="blast",
                     cfl=cfl, steps=rng.randint(3, 10))
    members = [log(2, 6 if p == 3 else 8) for _ in range(rng.randint(1, 4))]
    return _case(kind="batch", members=",".join(str(b) for b in members), B=max(members), p=p,
                 initial=rng.choice(["vortex", "smooth"]), cfl=cfl, steps=rng.randint(3, 6))


# ----------------------------------------------------------------- lattices
def _rotations(d):
    """The proper signed axis permutations: local axis a runs along global axis
    perm[a] with sign sign[a]."""
    out = []
    for perm in itertools.permutations(range(d)):
        odd = sum(perm[i] > perm[j] for i in range(d) for j in range(i + 1, d)) % 2
        for sign in itertools.product((1, -1), repeat=d):
            if math.prod(sign) == (-1 if odd else 1):
                out.append((perm, sign))
    return out


class Mesh:
    """Leaf blocks of a refined root lattice: (root, level, local position) in
    canonical order (root by root, depth first), their global positions and
    frames."""

    def __init__(self, case, B=None):
        self.d, self.n, self.B = case["dim"], case["n_seg"], case["B"] if B is None else B
        self.extent = case["extent"]
        d, n, B = self.d, self.n, self.B
        rng = np.random.default_rng(7)  # the mesh belongs to the case, not to a seed's state
        self.roots = [tuple((r // B ** a) % B for a in range(d)) for r in range(B ** d)]
        rots = _rotations(d)
        self.frames = [rots[int(rng.integers(len(rots)))] if case["rotate"] else (tuple(range(d)), (1,) * d)
                       for _ in self.roots]
        self.jitter = case["jitter"]
        self.lat = None
        if self.jitter > 0:
            h = self.extent / (B * n)
            lat = np.stack(np.meshgrid(*[h * np.arange(B * n + 1)] * d, indexing="ij"), -1)
            inner = (slice(1, -1),) * d
            lat[inner] += rng.uniform(-self.jitter * h, self.jitter * h, size=lat[inner].shape)
            self.lat = lat
        self.refined = set()  # (level, global position) of refined blocks
        self.rounds = []      # refined blocks, level by level
        for level in range(1, 4):
            want = [q for q in self._blocks(level) if self._wanted(case["refine"], level, q)]
            for q in want:
                self._refine(level, q)
        for level in range(1, 4):
            got = [q for (lv, q) in self.refined if lv == level]
            if got:
                self.rounds.append((level, got))
        self._enumerate()

    def _blocks(self, level):
        if level == 1:
            return list(self.roots)
        d = self.d
        return [tuple(2 * q[a] + (c >> a & 1) for a in range(d)) for (lv, q) in sorted(self.refined) if lv == level - 1
                for c in range(2 ** d)]

    def _wanted(self, rule, level, q):
        size = 1.0 / (self.B * 2 ** (level - 1))  # block edge over the domain's
        lo = [x * size for x in q]
        mid = [x + size / 2 for x in lo]
        if rule == "centre":  # the central half, once
            return level == 1 and all(0.25 <= m <= 0.75 for m in mid)
        if rule == "twice_centre":  # everything once, then one block below the centre
            return level == 1 or (level == 2 and all(x < 0.5 <= x + size + 1e-12 for x in lo))
        if rule in ("shell", "shell2"):  # the blocks that a sphere around the centre cuts
            near = math.sqrt(sum(max(x - 0.5, 0.0, 0.5 - x - size) ** 2 for x in lo))
            far = math.sqrt(sum(max(abs(x - 0.5), abs(x + size - 0.5)) ** 2 for x in lo))
            return level <= (2 if rule == "shell" else 1) and near <= 0.18 <= far
        return False

    def _refine(self, level, q):
        if (level, q) in self.refined:
            return
        if level > 1:
            self._refine(level - 1, tuple(x // 2 for x in q))
            m = self.B * 2 ** (level - 1)
            for a in range(self.d):  # at most one level between face neighbours
                for s in (-1, 1):
                    nb = tuple((x + s * (b == a)) % m for b, x in enumerate(q))
                    self._refine(level - 1, tuple(x // 2 for x in nb))
        self.refined.add((level, q))

    def _local(self, root, level, q):
        """Local position in the root's frame of the block at global position q."""
        perm, sign = self.frames[root]
        m = 2 ** (level - 1)
        out = []
        for a in range(self.d):
            x = q[perm[a]] - self.roots[root][perm[a]] * m
            out.append(x if sign[a] > 0 else m - 1 - x)
        return tuple(out)

    def _key(self, level, q):
        m, B = 2 ** (level - 1), self.B
        root = sum((q[a] // m) * B ** a for a in range(self.d))
        pos = self._local(root, level, q)
        path = tuple(sum((x >> (level - 2 - k) & 1) << a for a, x in enumerate(pos)) for k in range(level - 1))
        return root, path

    def _enumerate(self):
        leaves, todo = [], [(1, q) for q in self.roots]
        while todo:
            level, q = todo.pop()
            if (level, q) in self.refined:
                todo += [(level + 1, tuple(2 * q[a] + (c >> a & 1) for a in range(self.d))) for c in range(2 ** self.d)]
            else:
                leaves.append((self._key(level, q), level, q))
        leaves.sort()
        self.leaves = [(level, q) for _, level, q in leaves]
        self.index = {lq: i for i, lq in enumerate(self.leaves)}
        self.leaf_frame = [self.frames[k[0]] for k, _, _ in leaves]

    def with_refined(self, level, blocks):
        """This mesh with some of its leaves refined."""
        m = object.__new__(Mesh)
        m.__dict__.update(self.__dict__)
        m.refined = self.refined | {(level, q) for q in blocks}
        m._enumerate()
        return m

    def root_nodes(self):
        """Root corner nodes, corner ids and (jittered) cell nodes in local order."""
        d, n, B = self.d, self.n, self.B
        C = B + 1
        grid = np.stack(np.meshgrid(*[np.arange(C)] * d, indexing="ij"), -1).reshape(-1, d)
        order = np.argsort(sum(grid[:, a] * C ** a for a in range(d)))
        grid = grid[order]
        nodes = self.lat[tuple((grid * n).T)] if self.lat is not None else grid * (self.extent / B)
        corners, cells = [], [] if self.lat is not None else None
        k = np.arange(2 ** d)
        li = np.arange((n + 1) ** d)
        for root, b in enumerate(self.roots):
            perm, sign = self.frames[root]
            ids, g = 0, [None] * d
            for a in range(d):
                bit, I = k >> a & 1, (li // (n + 1) ** a) % (n + 1)
                ids = ids + (b[perm[a]] + (bit if sign[a] > 0 else 1 - bit)) * C ** perm[a]
                g[perm[a]] = b[perm[a]] * n + (I if sign[a] > 0 else n - I)
            corners.append(ids)
            if cells is not None:
                cells.append(self.lat[tuple(g)])
        return nodes, np.asarray(corners), None if cells is None else np.asarray(cells)

    def forest(self, case):
        nodes, corners, cells = self.root_nodes()
        periodic = [tuple(self.extent * (a == b) for b in range(self.d)) for a in range(self.d)]
        f = dgf.Forest(self.d, self.n, case["p"], nodes, corners, cells, periodic, precision=PRECISION[case["precision"]],
                       cfl=case["cfl"], nonconforming=case["nonconforming"])
        part = object.__new__(Mesh)
        part.__dict__.update(self.__dict__)
        part.refined = set()
        for level, blocks in self.rounds:
            part._enumerate()
            f.refine(sorted(part.index[(level, q)] for q in blocks))
            part.refined = part.refined | {(level, q) for q in blocks}
        assert f.n_leaves == len(self.leaves)
        if case["limiter"] > 0:
            f.set_limiter(case["limiter"])
        return f


# ------------------------------------------------- state arrays, global frame
# (leaf, variable, q_{d-1} .. q_0, cell_{d-1} .. cell_0); q: Gauss point
def _gauss(N):
    x, w = np.polynomial.legendre.leggauss(N)
    return x, w


def _legendre(N, x):
    return np.stack([np.polynomial.legendre.legval(x, np.eye(N)[k]) for k in range(N)], -1)


def _lagrange(N, x):
    """l_j(x_i) of the Gauss points' Lagrange basis."""
    return _legendre(N, np.asarray(x)) @ np.linalg.inv(_legendre(N, _gauss(N)[0]))


def _along(A, u, dim):
    """sum_j A[i][j] u_j along a dimension of u."""
    A = torch.as_tensor(A, dtype=torch.float64)
    parts = u.unbind(dim)
    return torch.stack([sum(float(A[i, j]) * parts[j] for j in range(len(parts))) for i in range(A.shape[0])], dim)


class Space:
    """Gauss points and metric of a mesh in the global frame."""

    def __init__(self, mesh, p, dev):
        self.m, self.N, self.dev = mesh, p + 1, dev
        self.d, self.n = mesh.d, mesh.n
        self.x, self.w = _gauss(self.N)
        self.scale = torch.tensor([2.0 ** (lv - 1) for lv, _ in mesh.leaves], dtype=torch.float64, device=dev)
        self.pos = torch.tensor([q for _, q in mesh.leaves], device=dev)
        self._node = None

    def qdim(self, a):
        return 2 + self.d - 1 - a

    def cdim(self, a):
        return 2 + 2 * self.d - 1 - a

    def _vec(self, v, a, at):
        """v laid along axis a of the point (at = 0) or cell (at = 1) dimensions."""
        s = [1] * (2 * self.d)
        s[(at + 1) * self.d - 1 - a] = len(v)
        return torch.as_tensor(np.asarray(v), dtype=torch.float64, device=self.dev).view(1, *s)

    def _corner(self, bits):
        """Positions of a corner of every cell: (leaf, component, 1.., cells)."""
        if self._node is None:
            d, n, B = self.d, self.n, self.m.B
            lat = torch.as_tensor(self.m.lat, dtype=torch.float64, device=self.dev)
            scale = self.scale.view(-1, 1)
            base, frac = [], []
            for a in range(d):
                s = (self.pos[:, a:a + 1] * n + torch.arange(n + 1, device=self.dev)) / scale
                lo = torch.clamp(torch.floor(s).long(), max=B * n - 1)
                base.append(lo)
                frac.append(s - lo)
            shape = lambda t, a: t.view(t.shape[0], *[n + 1 if b == a else 1 for b in reversed(range(d))])  # noqa: E731
            X = 0
            for c in range(2 ** d):
                w, idx = 1.0, []
                for a in range(d):
                    bit = c >> a & 1
                    w = w * (shape(frac[a], a) if bit else 1 - shape(frac[a], a))
                    idx.append(shape(base[a], a) + bit)
                X = X + w.unsqueeze(-1) * lat[tuple(idx)]
            self._node = X.movedim(-1, 1)
        sl = tuple(slice(b, b + self.n) for b in reversed(bits))
        X = self._node[(slice(None), slice(None)) + sl]
        return X.reshape(X.shape[0], X.shape[1], *[1] * self.d, *X.shape[2:])

    def points(self, leaves=slice(None)):
        """Physical Gauss points, one (leaf, q.., cell..) array per component."""
        d = self.d
        if self.m.jitter > 0:
            out = [0.0] * d
            for c in range(2 ** d):
                bits = [c >> a & 1 for a in range(d)]
                w = 1.0
                for a in range(d):
                    w = w * self._vec(0.5 * (1 + (2 * bits[a] - 1) * self.x), a, 0)
                X = self._corner(bits)[leaves]
                out = [out[j] + w * X[:, j] for j in range(d)]
            return out
        out = []
        scale, pos = self.scale[leaves], self.pos[leaves]
        for a in range(d):
            h = (self.m.extent / (self.m.B * scale * self.n)).view(-1, *[1] * (2 * d))
            i = pos[:, a].view(-1, *[1] * (2 * d)) * self.n + self._vec(np.arange(self.n), a, 1)
            t = h * (i + self._vec(0.5 * (1 + self.x), a, 0))
            out.append(t.expand(-1, *[self.N] * d, *[self.n] * d))
        return out

    def metric(self, a, at=None):
        """J grad xi_a at the Gauss points, or on the faces xi_a = at; and J."""
        d = self.d
        if self.m.jitter == 0:
            h = (0.5 * self.m.extent / (self.m.B * self.scale * self.n)).view(-1, *[1] * (2 * d))
            return [h ** (d - 1) if j == a else 0.0 * h for j in range(d)], h ** d
        t = [[0.0] * d for _ in range(d)]
        for c in range(2 ** d):
            bits = [c >> b & 1 for b in range(d)]
            X = self._corner(bits)
            for b in range(d):
                w = 0.5 * (2 * bits[b] - 1)
                for e in range(d):
                    if e != b:
                        xe = np.array([at]) if at is not None and e == a else self.x
                        w = w * self._vec(0.5 * (1 + (2 * bits[e] - 1) * xe), e, 0)
                for j in range(d):
                    t[b][j] = t[b][j] + w * X[:, j]
        if d == 2:
            row = [t[1][1], -t[1][0]] if a == 0 else [-t[0][1], t[0][0]]
        else:
            u, v = t[(a + 1) % 3], t[(a + 2) % 3]
            row = [u[(j + 1) % 3] * v[(j + 2) % 3] - u[(j + 2) % 3] * v[(j + 1) % 3] for j in range(3)]
        return row, sum(t[a][j] * row[j] for j in range(d))

    # modal arrays of the library: (leaf, variable, mode, cell), local frames
    def to_local(self, u):
        return self._frames(u, True)

    def to_global(self, u):
        return self._frames(u, False)

    def _frames(self, u, local):
        d, out = self.d, None
        groups = {}
        for i, fr in enumerate(self.m.leaf_frame):
            groups.setdefault(fr, []).append(i)
        if len(groups) == 1 and next(iter(groups)) == (tuple(range(d)), (1,) * d):
            return u
        out = torch.empty_like(u)
        for (perm, sign), ids in groups.items():
            ids = torch.tensor(ids, device=u.device)
            v = u[ids]
            src, flips = [0, 1] + [0] * (2 * d), []
            for a in range(d):
                l, g = a, perm[a]
                for dim in (self.qdim, self.cdim):
                    if local:
                        src[dim(l)] = dim(g)
                    else:
                        src[dim(g)] = dim(l)
                    if sign[a] < 0:
                        flips.append(dim(l) if local else dim(g))
            v = v.permute(src)
            out[ids] = v.flip(flips) if flips else v
        return out

    def modal(self, u):
        """Global nodal values -> modal coefficients in the library's layout."""
        u = self.to_local(u)
        V = np.linalg.inv(_legendre(self.N, self.x))
        for a in range(self.d):
            u = _along(V, u, self.qdim(a))
        return u.reshape(u.shape[0], u.shape[1], self.N ** self.d, self.n ** self.d)

    def nodal(self, K):
        u = K.double().view(K.shape[0], K.shape[1], *[self.N] * self.d, *[self.n] * self.d)
        V = _legendre(self.N, self.x)
        for a in range(self.d):
            u = _along(V, u, self.qdim(a))
        return self.to_global(u)


# ------------------------------------------------------------ initial states
def _initial(case, space, seed):
    """Modal state of a case for a seed (the library's element type)."""
    rng = np.random.default_rng(seed)
    d, L = case["dim"], len(space.m.leaves)
    offs, phase = rng.uniform(-1, 1, 3), rng.uniform(0, 2 * math.pi, 4)
    amp = rng.uniform(0.8, 1.0)
    out_t = torch.float32 if case["precision"] == "fp32" else torch.float64
    K = torch.empty((L, d + 2, (case["p"] + 1) ** d, case["n_seg"] ** d), dtype=out_t, device=space.dev)
    size = max(1, (1 << 25) // ((case["p"] + 1) ** d * case["n_seg"] ** d))
    rotated = any(f != space.m.leaf_frame[0] for f in space.m.leaf_frame)
    size = L if rotated else size
    V = np.linalg.inv(_legendre(space.N, space.x))
    for lo in range(0, L, size):
        x = space.points(slice(lo, lo + size))
        e = space.m.extent
        if case["initial"] == "vortex":
            s = 10.0 / e
            X = [torch.remainder(s * x[a] - (5.0 + 2.0 * offs[a]) + 5.0, 10.0) - 5.0 for a in range(2)]
            beta = 5.0 * amp
            g = torch.exp(0.5 * (1.0 - X[0] ** 2 - X[1] ** 2))
            T = 1.0 - (GAMMA - 1) * beta ** 2 / (8 * GAMMA * math.pi ** 2) * g * g
            rho = T ** (1 / (GAMMA - 1))
            vel = [1.0 - beta / (2 * math.pi) * g * X[1], 1.0 + beta / (2 * math.pi) * g * X[0]] + [torch.ones_like(T)] * (d - 2)
            pr = rho ** GAMMA
        elif case["initial"] == "blast":
            h = e / (case["B"] * case["n_seg"] * 2.0)
            r = torch.sqrt(sum((x[a] / e - 0.5 - 0.01 * offs[a]) ** 2 for a in range(d)))
            s = 0.5 * (1 - torch.tanh((r - 0.18) * e / (2.0 * h)))
            rho, pr, vel = 1 + 7 * amp * s, 1 + 9 * amp * s, [torch.zeros_like(r)] * d
        else:
            w = [2 * math.pi * x[a] / e for a in range(d)]
            rho = 1 + 0.2 * amp * math.prod([torch.sin(t + phase[0]) for t in w]) + 0.1 * torch.cos(w[0] + phase[1])
            vel = [0.3 + 0.1 * torch.cos(t + phase[2]) for t in w]
            pr = 1 + 0.1 * torch.sin(sum(w) + phase[3])
        u = torch.stack([rho] + [rho * v for v in vel] + [pr / (GAMMA - 1) + 0.5 * rho * sum(v * v for v in vel)], 1)
        if rotated:
            K.copy_(space.modal(u))
        else:
            for a in range(d):
                u = _along(V, u, space.qdim(a))
            K[lo:lo + size] = u.reshape(u.shape[0], d + 2, K.shape[2], K.shape[3])
    return K


def _meshes(case):
    if case["kind"] == "batch":
        return [Mesh(case, int(b)) for b in case["members"].split(",")]
    return [Mesh(case)]


def _cycle_blocks(mesh):
    """Root blocks that an adaptive cycle refines and coarsens again: every
    third of the unrefined ones whose neighbours allow it."""
    return [q for (lv, q) in mesh.leaves if lv == 1][::3]


# ------------------------------------------------------------ the user's calls
def prepare(case, seed):
    dev = torch.device("cuda")
    state = dict(case=case, forests=[], U=[], out=[])
    for i, mesh in enumerate(_meshes(case)):
        c = dict(case, B=mesh.B)
        f = mesh.forest(c)
        U = _initial(c, Space(mesh, case["p"], dev), seed + 1000 * i)
        state["forests"].append(f)
        state["U"].append(U)
        state["out"].append(torch.empty_like(U))
    if case["kind"] == "batch":
        state["batch"] = dgf.Batch()
    if case["kind"] == "cycle":
        mesh = _meshes(case)[0]
        blocks = set(_cycle_blocks(mesh))
        fine = mesh.with_refined(1, blocks)
        state["refine"] = np.array([float(lv == 1 and q in blocks) for lv, q in mesh.leaves]) + 0.5
        state["coarsen"] = np.array([0.0 if lv == 2 and tuple(x // 2 for x in q) in blocks else 0.5
                                     for lv, q in fine.leaves])
    torch.cuda.synchronize()
    return state


def run(state):
    case, steps = state["case"], state["case"]["steps"]
    forests, U, out = state["forests"], state["U"], state["out"]
    if case["kind"] == "batch":
        b = state["batch"]
        for f, u in zip(forests, U):
            f.set_state(u)
        b.set(forests, [math.inf] * len(forests))
        b.step(steps)
        _, _, status = b.progress()
        return {"state": [f.get_state(o) for f, o in zip(forests, out)], "status": status}
    f = forests[0]
    f.set_state(U[0])
    for _ in range(steps):
        f.rk_step()
    if case["kind"] == "cycle":
        marked = f.indicator()
        f.adapt(1.0, 0.25, 2, indicator=state["refine"])
        leaves = f.n_leaves
        for _ in range(steps):
            f.rk_step()
        f.adapt(1.0, 0.25, 2, indicator=state["coarsen"])
        return {"state": f.get_state(out[0]), "indicator": marked, "leaves": leaves}
    return {"state": f.get_state(out[0])}


def work(case):
    """State values read and written and floating-point operations of one pass."""
    d, N, n, nv = case["dim"], case["p"] + 1, case["n_seg"], case["dim"] + 2
    size = 4 if case["precision"] == "fp32" else 8
    cells = sum(len(m.leaves) for m in _meshes(case)) * n ** d
    points = cells * N ** d
    stages = 3 * case["steps"] * (2 if case["kind"] == "cycle" else 1)
    # a stage reads its input and (stages 2, 3) U^n and writes its output; the
    # state is handed over and read back once
    values = points * nv * (8 / 3 * stages + 4)
    # per point and direction: the flux, the derivative and two lifts of nv
    # variables; per face point one Lax-Friedrichs flux and two traces
    flux, faces = 4 * d + 3 * nv + 6, cells * d * N ** (d - 1)
    flops = stages * (points * (d * (flux + nv * (2 * N + 4)) + 6 * nv) + faces * (2 * flux + 8 * nv + 4 * N * nv))
    return {"bytes": values * size, "flops": flops}


# ---------------------------------------------------------------- FP64 solver
def _pressure(u):
    ke = sum(u[k] * u[k] for k in range(1, len(u) - 1))
    return (GAMMA - 1) * (u[-1] - 0.5 * ke / u[0])


def _flux(u, row):
    vn = sum(u[1 + j] * row[j] for j in range(len(row))) / u[0]
    p = _pressure(u)
    return [u[0] * vn] + [u[1 + j] * vn + p * row[j] for j in range(len(row))] + [(u[-1] + p) * vn], vn, p


def _lax_friedrichs(uL, uR, row):
    FL, vL, pL = _flux(uL, row)
    FR, vR, pR = _flux(uR, row)
    area = torch.sqrt(sum(r * r for r in row))
    al = torch.maximum(vL.abs() + torch.sqrt(GAMMA * pL / uL[0]) * area, vR.abs() + torch.sqrt(GAMMA * pR / uR[0]) * area)
    return [0.5 * (a + b + al * (l - r)) for a, b, l, r in zip(FL, FR, uL, uR)]


class Solver:
    """SSP-RK3 of the DG residual on the global nodal state (all in FP64)."""

    def __init__(self, case, mesh, dev):
        self.case, self.s = case, Space(mesh, case["p"], dev)
        s, N, d = self.s, case["p"] + 1, case["dim"]
        self.d, self.N, self.n, self.dev = d, N, case["n_seg"], dev
        l = _lagrange(N, [-1.0, 1.0])
        self.lm, self.lp = l[0], l[1]
        V = _legendre(N, s.x)
        dV = np.stack([np.polynomial.legendre.legval(s.x, np.polynomial.legendre.legder(np.eye(N)[k])) if N > 1
                       else np.zeros(N) for k in range(N)], -1)
        D = dV @ np.linalg.inv(V)  # D[j][q] = l_q'(x_j)
        self.Sh = (D.T * s.w[None, :]) / s.w[:, None]
        self.split = [_lagrange(N, 0.5 * (s.x + e)) for e in (-1, 1)]  # to the lower, upper child
        self.weight = 1.0
        for a in range(d):
            self.weight = self.weight * s._vec(s.w, a, 0)
        self.h = (self.weight * s.metric(0)[1]).sum(tuple(range(1, 1 + d)), keepdim=True) ** (1.0 / d)
        self._neighbours()

    def _neighbours(self):
        """Per face: same-level pairs, coarser neighbours, finer neighbours."""
        m, d = self.s.m, self.d
        self.same, self.coarser, self.finer = {}, {}, {}
        for f in range(2 * d):
            a, sd = f >> 1, 2 * (f & 1) - 1
            same, coarser, finer = [], [], []
            for i, (lv, q) in enumerate(m.leaves):
                M = m.B * 2 ** (lv - 1)
                nb = tuple((x + sd * (b == a)) % M for b, x in enumerate(q))
                j = m.index.get((lv, nb))
                if j is not None:
                    same.append((i, j))
                    continue
                j = m.index.get((lv - 1, tuple(x // 2 for x in nb))) if lv > 1 else None
                if j is not None:
                    coarser.append((i, j))
                    continue
                tang = [b for b in range(d) if b != a]
                kids = []
                for c in range(2 ** (d - 1)):
                    k = [2 * x for x in nb]
                    k[a] += 0 if sd > 0 else 1
                    for t, b in enumerate(tang):
                        k[b] += c >> t & 1
                    kids.append(m.index[(lv + 1, tuple(k))])
                finer.append((i, kids))
            self.same[f], self.coarser[f], self.finer[f] = same, coarser, finer

    def _long(self, v):
        return torch.tensor(v, device=self.dev, dtype=torch.long)

    def trace(self, u, a, side):
        w = self.lp if side else self.lm
        return sum(float(w[k]) * u.select(self.s.qdim(a), k) for k in range(self.N)).unsqueeze(self.s.qdim(a))

    def _gather_fine(self, v, a, side, kids):
        """Fine blocks of a face as one array over the coarse guard cells: a
        leading child index e (bits over all axes), cells over the tangential
        axes; v holds (leaf, ..., cells)."""
        d, n, nd = self.d, self.n, v.dim()
        cd = lambda b: nd - 1 - b  # noqa: E731
        tang = [b for b in range(d) if b != a]
        halves = [v[self._long([k[c] for k in kids])] for c in range(2 ** (d - 1))]
        for t in range(len(tang)):  # join the sub-blocks along each tangential axis, lowest first
            halves = [torch.cat([halves[c], halves[c + 1]], cd(tang[t])) for c in range(0, len(halves), 2)]
        w = halves[0]  # 2n cells along the tangential axes, n along a
        out = []
        for e in range(2 ** d):
            z = w
            for b in range(d):
                bit = e >> b & 1
                if b == a:  # the two layers next to the face
                    k = bit if side else n - 2 + bit
                    z = z.narrow(cd(b), k, 1)
                else:
                    idx = torch.arange(bit, 2 * n, 2, device=v.device)
                    z = z.index_select(cd(b), idx)
            out.append(z)
        return out

    def _combine(self, u, J):
        """J-weighted projection of the 2^d children's nodal values u[e], J[e]
        (.., q.., cells..) onto the parent's Gauss points."""
        d, N, Q = self.d, self.N, self.N ** self.d
        flat = lambda t: t.flatten(-2 * d, -d - 1).movedim(-d - 1, -1)  # noqa: E731  (.., cells.., Q)
        M, rhs = 0.0, 0.0
        full = [J[0].shape[0], 1] + [N] * d
        for e in range(2 ** d):
            P = torch.ones((1, 1), dtype=torch.float64, device=self.dev)
            for a in reversed(range(d)):
                P = torch.kron(P, torch.as_tensor(self.split[e >> a & 1], device=self.dev))
            wj = (self.weight * J[e]).unsqueeze(1)
            wj = flat(wj.expand(*full, *wj.shape[-d:]))
            M = M + torch.einsum("...q,qk,ql->...kl", wj, P, P)
            rhs = rhs + torch.einsum("...q,qk->...k", wj * flat(u[e]), P)
        c = torch.linalg.solve(M, rhs.unsqueeze(-1)).squeeze(-1)
        return c.movedim(-1, -d - 1).unflatten(-d - 1, (N,) * d)

    def guard(self, u, f):
        """Traces that the blocks see across their face f: (leaf, variable,
        q.., 1 cell along the axis)."""
        s, d, n, N = self.s, self.d, self.n, self.N
        a, side = f >> 1, f & 1
        # neighbours are seen through their opposite face
        layer = u.narrow(s.cdim(a), 0 if side else n - 1, 1)
        tr = self.trace(layer, a, 1 - side)
        out = torch.empty_like(tr)
        if self.same[f]:
            i, j = zip(*self.same[f])
            out[self._long(i)] = tr[self._long(j)]
        tang = [b for b in range(d) if b != a]
        for i, j in self.coarser[f]:
            t = tr[j:j + 1]
            for b in tang:
                half = s.m.leaves[i][1][b] & 1
                t = t.narrow(s.cdim(b), half * (n // 2), n // 2)
                lo, up = (_along(self.split[e], t, s.qdim(b)) for e in (0, 1))
                t = torch.stack([lo, up], s.cdim(b) + 1).flatten(s.cdim(b), s.cdim(b) + 1)
            out[i] = t[0]
        if self.finer[f]:
            i, kids = zip(*self.finer[f])
            J = s.metric(a)[1].expand(len(s.m.leaves), *[N] * d, *[n] * d)
            g = self._combine(self._gather_fine(u, a, side, kids), self._gather_fine(J, a, side, kids))
            out[self._long(i)] = self.trace(g, a, 1 - side)
        return out

    def _mortar(self, a, side, F):
        """Coarse faces take the fine side's fluxes, tested with their own basis."""
        s, d, n, N = self.s, self.d, self.n, self.N
        f = 2 * a + side
        if not self.finer[f]:
            return
        i, kids = zip(*self.finer[f])
        tang = [b for b in range(d) if b != a]
        # fluxes on the fine blocks' opposite face, as (leaf, v, q.., 1, cells..)
        v = F.narrow(s.cdim(a), 0 if side else n, 1)
        halves = [v[self._long([k[c] for k in kids])] for c in range(2 ** (d - 1))]
        for b in tang:
            halves = [torch.cat([halves[c], halves[c + 1]], s.cdim(b)) for c in range(0, len(halves), 2)]
        w = halves[0]
        for b in tang:
            lift = [(self.split[e].T * s.w[None, :]) / s.w[:, None] for e in (0, 1)]
            w = sum(_along(lift[e], w.index_select(s.cdim(b), torch.arange(e, 2 * n, 2, device=self.dev)), s.qdim(b))
                    for e in (0, 1))
        idx = self._long(i)
        k = n if side else 0
        G = F.narrow(s.cdim(a), k, 1)
        G[idx] = w

    def residual(self, u):
        s, d = self.s, self.d
        R = torch.zeros_like(u)
        var = lambda t: list(t.unbind(1))  # noqa: E731
        for a in range(d):
            tm, tp = self.trace(u, a, 0), self.trace(u, a, 1)
            uL = torch.cat([self.guard(u, 2 * a), tp], s.cdim(a))
            uR = torch.cat([tm, self.guard(u, 2 * a + 1)], s.cdim(a))
            row, _ = s.metric(a, -1.0)
            if s.m.jitter > 0:
                last, _ = s.metric(a, 1.0)
                row = [torch.cat([r, l.narrow(s.cdim(a) - 1, self.n - 1, 1)], s.cdim(a) - 1) for r, l in zip(row, last)]
            F = torch.stack(_lax_friedrichs(var(uL), var(uR), row), 1)
            del uL, uR
            if self.case["nonconforming"] == "mortar":
                for side in (0, 1):
                    self._mortar(a, side, F)
            lo, up = F.narrow(s.cdim(a), 0, self.n), F.narrow(s.cdim(a), 1, self.n)
            G = torch.stack(_flux(var(u), s.metric(a)[0])[0], 1)
            R += _along(self.Sh, G, s.qdim(a))
            R += s._vec(self.lm / s.w, a, 0).unsqueeze(1) * lo - s._vec(self.lp / s.w, a, 0).unsqueeze(1) * up
        return R / s.metric(0)[1].unsqueeze(1)

    def dt(self, u):
        v = u.unbind(1)
        c = torch.sqrt(GAMMA * _pressure(v) / v[0])
        lam = sum((v[1 + j] / v[0]).abs() + c for j in range(self.d))
        return self.case["cfl"] * float((self.h / lam).min())

    def limit(self, u):
        """Scaling toward the cell mean that keeps density and pressure above
        the limiter's bound at every volume and face Gauss point."""
        eps, s, d = self.case["limiter"], self.s, self.d
        if eps == 0:
            return u
        qd = tuple(range(2, 2 + d))
        wj = (self.weight * s.metric(0)[1]).unsqueeze(1)
        mean = (wj * u).sum(qd, keepdim=True) / (wj * torch.ones_like(u[:, :1])).sum(qd, keepdim=True)
        pbar = _pressure(mean.unbind(1)).unsqueeze(1)
        chk = [u.flatten(2, 1 + d)]
        for a in range(d):
            chk += [self.trace(u, a, side).flatten(2, 1 + d) for side in (0, 1)]
        x, mb = torch.cat(chk, 2), mean.flatten(2, 1 + d)
        pb = pbar.flatten(2, 1 + d)
        rmin = x[:, :1].amin(2, keepdim=True)
        r0 = mb[:, :1]
        th1 = torch.where(rmin >= eps * r0, torch.ones_like(rmin), ((1 - eps) * r0 / (r0 - rmin)).clamp(max=1.0))
        du = th1 * (x - mb)
        low = _pressure((mb + du).unbind(1)).unsqueeze(1) < eps * pb
        # (E - eps p/(gamma-1)) rho = |m|^2 / 2 along the segment: a t^2 + b t + c = 0
        Eb = mb[:, -1:] - eps * pb / (GAMMA - 1)
        dm, mm = du[:, 1:-1], mb[:, 1:-1]
        A = du[:, -1:] * du[:, :1] - 0.5 * (dm * dm).sum(1, keepdim=True)
        Bq = Eb * du[:, :1] + du[:, -1:] * r0 - (mm * dm).sum(1, keepdim=True)
        C = Eb * r0 - 0.5 * (mm * mm).sum(1, keepdim=True)
        disc = torch.sqrt((Bq * Bq - 4 * A * C).clamp(min=0.0))
        # the smallest root in [0, 1], written so that it does not cancel
        den = -Bq + torch.where(Bq < 0, disc, -disc)
        roots = [2 * C / den, den / (2 * A)]
        t = torch.full_like(A, 2.0)
        for r in roots:
            t = torch.where((r >= 0) & (r <= 1) & (r < t), r, t)
        t = torch.where(t > 1, torch.zeros_like(t), t)
        th2 = torch.where(low, t, torch.ones_like(t)).amin(2, keepdim=True)
        th = (th1 * th2).view(u.shape[0], 1, *[1] * d, *u.shape[2 + d:])
        return mean + th * (u - mean)

    def march(self, u, steps):
        for _ in range(steps):
            dt = self.dt(u)
            v = self.limit(u + dt * self.residual(u))
            v = self.limit(0.75 * u + 0.25 * (v + dt * self.residual(v)))
            u = self.limit(u / 3 + 2 / 3 * (v + dt * self.residual(v)))
        return u

    def indicator(self, u):
        V = np.linalg.inv(_legendre(self.N, self.s.x))
        K = u[:, :1]
        for a in range(self.d):
            K = _along(V, K, self.s.qdim(a))
        first = lambda a: K[(slice(None), 0) + tuple(int(b == a) for b in reversed(range(self.d)))]  # noqa: E731
        mean = K[(slice(None), 0) + (0,) * self.d]
        return (2 * torch.sqrt(sum(first(a) ** 2 for a in range(self.d))) / mean).flatten(1).amax(1)


def _transfer(coarse, fine, u, blocks):
    """State of the mesh with the blocks refined (their parents split)."""
    s, d, n = fine.s, fine.d, fine.n
    out = torch.empty((len(fine.s.m.leaves),) + u.shape[1:], dtype=u.dtype, device=u.device)
    for i, (lv, q) in enumerate(s.m.leaves):
        j = coarse.s.m.index.get((lv, q))
        if j is not None:
            out[i] = u[j]
            continue
        t = u[coarse.s.m.index[(lv - 1, tuple(x // 2 for x in q))]].unsqueeze(0)
        for b in range(d):
            t = t.narrow(s.cdim(b), (q[b] & 1) * (n // 2), n // 2)
            t = torch.stack([_along(fine.split[e], t, s.qdim(b)) for e in (0, 1)], s.cdim(b) + 1).flatten(s.cdim(b), s.cdim(b) + 1)
        out[i] = t[0]
    return out


def _restrict(coarse, fine, v, blocks):
    """State of the coarse mesh from the refined one (children combined)."""
    s, d, n = coarse.s, coarse.d, coarse.n
    out = torch.empty((len(s.m.leaves),) + v.shape[1:], dtype=v.dtype, device=v.device)
    Jf = fine.s.metric(0)[1].expand(len(fine.s.m.leaves), *[coarse.N] * d, *[n] * d)
    for i, (lv, q) in enumerate(s.m.leaves):
        j = fine.s.m.index.get((lv, q))
        if j is not None:
            out[i] = v[j]
            continue
        kids = [fine.s.m.index[(lv + 1, tuple(2 * q[a] + (c >> a & 1) for a in range(d)))] for c in range(2 ** d)]

        def joined(t, first):
            parts = [t[k:k + 1] for k in kids]
            for b in range(d):
                parts = [torch.cat([parts[c], parts[c + 1]], t.dim() - 1 - b) for c in range(0, len(parts), 2)]
            kid = []
            for e in range(2 ** d):
                z = parts[0]
                for b in range(d):
                    z = z.index_select(z.dim() - 1 - b, torch.arange(e >> b & 1, 2 * n, 2, device=t.device))
                kid.append(z)
            return kid

        out[i] = coarse._combine(joined(v, 0), joined(Jf, 0))[0]
    return out


def exact(case, seed):
    """The outputs of ``run`` in FP64 on the same (rounded) inputs."""
    dev = torch.device("cuda")
    states = []
    for i, mesh in enumerate(_meshes(case)):
        c = dict(case, B=mesh.B)
        S = Solver(c, mesh, dev)
        u = S.s.nodal(_initial(c, S.s, seed + 1000 * i))
        u = S.march(u, case["steps"])
        if case["kind"] == "cycle":
            marked = S.indicator(u)
            blocks = _cycle_blocks(mesh)
            F = Solver(c, mesh.with_refined(1, blocks), dev)
            v = F.march(_transfer(S, F, u, blocks), case["steps"])
            u = _restrict(S, F, v, blocks)
            return {"state": S.s.modal(u), "indicator": marked.cpu().numpy(), "leaves": None}
        states.append(S.s.modal(u))
    if case["kind"] == "batch":
        return {"state": states, "status": None}
    return {"state": states[0]}
