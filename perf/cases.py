"""The work a user of this library has it do, as measured cases.

A case goes through the public entry points of the package: the factorisation,
the selected inversion in the schedule such a user picks, and the entries or
gradients that are read from it.  Matrices are the families of this
repository: 5- and 7-point grid operators, graph Laplacians with random edge
weights, upwind convection-diffusion (non-symmetric), shifted (indefinite)
grids, block-sparse Hamiltonians with complex poles, uneven batches of grids,
and dense blocks.  All are held as lower CSC in natural order with a nested
dissection ordering passed to the analysis.

A pass takes new values and does everything that depends on them: a program
analyses a pattern once and then factors and inverts for every new set of
values (a time step, a pole, an optimiser step).
"""
import functools
import math

import numpy as np
import torch

import paper_1404_0447_gb300 as P

# --------------------------------------------------------------------------
# patterns, orderings and values
# --------------------------------------------------------------------------


@functools.lru_cache(maxsize=64)
def _pattern(dims, nb):
    """Lower CSC of a box grid of elements with nb unknowns each, every element coupled to its face
    neighbours (nb = 1: the 5- or 7-point grid).  Entry order: per element e and column a the slots
    (e itself, then its +x, +y, +z neighbours) by rows; `keep` marks the stored entries of that
    [element, column, slot, row] array."""
    mx, my, mz = dims
    ne = mx * my * mz
    e = np.arange(ne)
    x, y, z = e % mx, e // mx % my, e // (mx * my)
    nbr = np.stack([e, e + 1, e + mx, e + mx * my], 1)
    have = np.stack([np.ones(ne, bool), x + 1 < mx, y + 1 < my, z + 1 < mz], 1)
    a = np.arange(nb)
    keep = np.broadcast_to(have[:, None, :, None], (ne, nb, 4, nb)).copy()
    keep[:, :, 0, :] = a[None, None, :] >= a[None, :, None]
    rows = np.broadcast_to((nbr * nb)[:, None, :, None] + a, (ne, nb, 4, nb))[keep].astype(np.int32)
    colptr = np.concatenate([[0], np.cumsum(keep.sum((2, 3)).ravel())]).astype(np.int64)
    return ne * nb, colptr, rows, nbr, have, keep


@functools.lru_cache(maxsize=64)
def _order(dims, nb):
    """Nested dissection of the element grid: a box of at most 8 elements (or thinner than 3) is numbered
    along its rows, any other is cut across its longest axis: left part, right part, the plane between."""
    mx, my, _ = dims
    out = []

    def rec(lo, hi):
        ext = [h - l for l, h in zip(lo, hi)]
        if min(ext) <= 0:
            return
        if math.prod(ext) <= 8 or max(ext) < 3:
            zz, yy, xx = np.meshgrid(*(np.arange(lo[i], hi[i]) for i in (2, 1, 0)), indexing="ij")
            out.append((xx + mx * (yy + my * zz)).ravel())
            return
        ax = ext.index(max(ext))
        c = lo[ax] + (ext[ax] - 1) // 2
        left, right, a, b = list(hi), list(lo), list(lo), list(hi)
        left[ax], right[ax], a[ax], b[ax] = c, c + 1, c, c + 1
        rec(lo, tuple(left))
        rec(tuple(right), hi)
        zz, yy, xx = np.meshgrid(*(np.arange(a[i], b[i]) for i in (2, 1, 0)), indexing="ij")
        out.append((xx + mx * (yy + my * zz)).ravel())

    rec((0, 0, 0), dims)
    perm = np.concatenate(out)
    return (perm[:, None] * nb + np.arange(nb)).ravel().astype(np.int32)


def _dims(case):
    d = [int(v) for v in str(case["dims"]).split("x")]
    return tuple(d + [1] * (3 - len(d)))


def _grid_values(dims, diag, off):
    """Lower-CSC values of a grid from its diagonal [n] and edge values [n, 3] (+x, +y, +z)."""
    _, _, _, _, _, keep = _pattern(dims, 1)
    v = np.concatenate([diag[:, None], off], 1)
    return v[keep[:, 0, :, 0]]


def _members(case):
    """Grid dimensions of an uneven batch: `squares` and `cubes` hold the sides."""
    sq = [int(v) for v in str(case["squares"]).split(",") if v]
    cu = [int(v) for v in str(case["cubes"]).split(",") if v]
    both = [(m, m, 1) for m in sq] + [(m, m, m) for m in cu]
    return sorted(both, key=lambda d: (d[0] * 7919 + d[2]) % 101)


def _pieces(case, seed):
    """The matrices of a case, each (dims, diag, lower edge values, upper edge values)."""
    g = np.random.default_rng(seed)
    kind = case["kind"]
    out = []
    for dims in _members(case) if kind == "uneven" else [_dims(case)] * int(case.get("batch", 1)):
        n, _, _, nbr, have, _ = _pattern(dims, 1)
        h = have[:, 1:]
        axes = sum(m > 1 for m in dims)
        if kind in ("logdet", "adjoint"):  # graph Laplacian: conductances exp(N(0, 1/4)), + 0.05 I
            w = np.where(h, np.exp(g.normal(0.0, 0.5, (n, 3))), 0.0)
            lo = up = -w
            diag = 0.05 + w.sum(1)
            np.add.at(diag, nbr[:, 1:][h], w[h])
        elif kind == "unsym":  # upwind convection-diffusion, diagonally dominant
            b = np.where(h, g.uniform(-0.5, 0.5, (n, 3)), 0.0)
            lo, up = np.where(h, -(1.0 + b), 0.0), np.where(h, -(1.0 - b), 0.0)
            w = np.where(h, 1.0 + np.abs(b), 0.0)
            diag = g.uniform(0.01, 0.1, n) + w.sum(1)
            np.add.at(diag, nbr[:, 1:][h], w[h])
        else:
            lo = up = np.where(h, -1.0, 0.0)
            if kind == "indefinite":  # the grid Laplacian shifted into its spectrum
                diag = 2.0 * axes - 0.5 + g.uniform(-0.05, 0.05, n)
            else:
                diag = 2.0 * axes + (g.uniform(0.01, 0.1, n) if axes == 3 and kind != "uneven" else g.uniform(0.1, 1.0, n))
        out.append((dims, diag, lo, up))
    return out


def _hamiltonian(case, seed):
    """Blocks [element, slot, row, column] of a DG-like Hamiltonian (diagonal blocks dominate) and its poles."""
    g = np.random.default_rng(seed)
    dims, nb, npoles = _dims(case), int(case["nb"]), int(case["poles"])
    ne = math.prod(dims)
    blocks = g.normal(0.0, 1.0, (ne, 4, nb, nb)) * (0.1 / math.sqrt(nb))
    d = g.normal(0.0, 1.0, (ne, nb, nb))
    blocks[:, 0] = (d + d.transpose(0, 2, 1)) / (2.0 * math.sqrt(nb)) + 2.0 * np.eye(nb)
    t = np.sort(g.uniform(0.0, np.pi, npoles))
    z = 0.5 * (1.0 + np.cos(t)) + 0.5j * np.sin(t)
    w = g.normal(0.0, 1.0, npoles) + 1j * g.normal(0.0, 1.0, npoles)
    return blocks, z, w


def _pole_values(case, blocks, z):
    dims, nb = _dims(case), int(case["nb"])
    _, colptr, _, _, _, keep = _pattern(dims, nb)
    hv = blocks.transpose(0, 3, 1, 2)[keep]
    v = np.repeat(hv[None].astype(np.complex128), len(z), 0)
    v[:, colptr[:-1]] -= z[:, None]
    return v


def _dense_blocks(case, seed):
    """Unit lower triangles and pivots of SPD blocks, as their L D L^T gives them (column-major)."""
    s, count = int(case["order"]), int(case["count"])
    g = torch.Generator().manual_seed(seed)
    a = torch.randn(count, s, s, generator=g, dtype=torch.float64)
    a = a @ a.transpose(1, 2) / s + torch.eye(s, dtype=torch.float64)
    c = torch.linalg.cholesky(a)
    d = torch.diagonal(c, dim1=1, dim2=2)
    return c / d[:, None, :], d * d


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------


def listed():
    return [
        # one small 2D problem, analysed with fundamental supernodes: the smallest call, all launches and latency
        dict(name="grid2d_31", kind="selinv", dims="31x31", batch=1, mode=P.LEVEL, relax=P.RELAX_NONE),
        # a 2D sheet of ragged sides, inverted again for every new diagonal through the captured schedule
        dict(name="grid2d_200x147_graph", kind="selinv", dims="200x147", batch=1, mode=P.GRAPH, relax=P.RELAX_AMALG),
        # many small systems of one pattern at once (a batch of shifts)
        dict(name="grid3d_12_batch16", kind="selinv", dims="12x12x12", batch=16, mode=P.GRAPH, relax=P.RELAX_AMALG),
        # an ordinary 3D problem of odd, unequal sides in the default schedule
        dict(name="grid3d_33x29x27", kind="selinv", dims="33x29x27", batch=1, mode=P.LEVEL, relax=P.RELAX_AMALG),
        # a large 3D problem: FEM-class selected inversion, bound by arithmetic
        dict(name="grid3d_56", kind="selinv", dims="56x56x56", batch=1, mode=P.LEVEL, relax=P.RELAX_AMALG),
        # maximum-likelihood training: log det of a graph Laplacian and its gradient, one optimiser step
        dict(name="logdet_24", kind="logdet", dims="24x24x24"),
        # a loss on marginal variances and neighbour covariances: selected inverse forward, its adjoint backward
        dict(name="adjoint_20", kind="adjoint", dims="20x20x20"),
        # pole expansion of a block-sparse Hamiltonian: complex symmetric batch with the pole sum
        dict(name="poles_4x4x4_nb48", kind="poles", dims="4x4x4", nb=48, poles=4),
        # independent 2D and 3D problems of uneven size in one persistent launch
        dict(name="uneven_10", kind="uneven", squares="64,97,131,160,211", cubes="16,17,20,23,25", mode=P.PERSISTENT),
        # transport problem: non-symmetric values on a symmetric pattern, both triangles of the inverse
        dict(name="convdiff_24", kind="unsym", dims="24x24x24", mode=P.LEVEL),
        # indefinite system with pivots inside the supernodes (density of states at a shift inside the spectrum)
        dict(name="indefinite_26x25x23", kind="indefinite", dims="26x25x23", mode=P.LEVEL),
        # dense diagonal blocks inverted inside another program's memory pool (block preconditioner)
        dict(name="blocks_100", kind="blocks", order=100, count=192),
    ]


def draw(rng):
    kind = rng.choice(["selinv2", "selinv2", "selinv3", "selinv3", "batch", "logdet", "adjoint", "poles", "uneven",
                       "unsym", "indefinite", "blocks"])
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    def near(m):
        return max(3, m + rng.randint(-m // 8, m // 8))
    mode = rng.choice([P.LEVEL, P.GRAPH, P.PERSISTENT])
    relax = rng.choice([P.RELAX_AMALG, P.RELAX_AMALG, P.RELAX_NONE])
    if kind == "selinv2":
        m = size(20, 360)
        return dict(kind="selinv", dims=f"{near(m)}x{near(m)}", batch=1, mode=mode, relax=relax)
    if kind == "selinv3":
        m = size(8, 46)
        return dict(kind="selinv", dims=f"{near(m)}x{near(m)}x{near(m)}", batch=1, mode=mode, relax=relax)
    if kind == "batch":
        m = size(6, 20)
        return dict(kind="selinv", dims=f"{near(m)}x{near(m)}x{near(m)}", batch=rng.randint(2, 16), mode=mode, relax=relax)
    if kind in ("logdet", "adjoint"):
        m = size(8, 28 if kind == "logdet" else 20)
        return dict(kind=kind, dims=f"{near(m)}x{near(m)}x{near(m)}")
    if kind == "poles":
        return dict(kind="poles", dims="x".join(str(rng.randint(2, 5)) for _ in range(3)), nb=rng.randint(6, 48),
                    poles=rng.randint(1, 8))
    if kind == "uneven":
        return dict(kind="uneven", squares=",".join(str(size(64, 256)) for _ in range(rng.randint(1, 6))),
                    cubes=",".join(str(rng.randint(16, 28)) for _ in range(rng.randint(1, 6))), mode=mode)
    if kind in ("unsym", "indefinite"):
        m = size(8, 28)
        mode = rng.choice([P.LEVEL, P.GRAPH])
        return dict(kind=kind, dims=f"{near(m)}x{near(m)}x{near(m)}", mode=mode)
    s = rng.randint(8, 128)
    return dict(kind="blocks", order=s, count=max(1, min(size(4, 1024), (1 << 21) // (s * s))))


# --------------------------------------------------------------------------
# a program's side of each case
# --------------------------------------------------------------------------


def _handle(case):
    kind = case["kind"]
    if kind == "uneven":
        pats = [_pattern(d, 1) for d in _members(case)]
        return P.SelInv([p[0] for p in pats], [p[1] for p in pats], [p[2] for p in pats],
                        perm=[_order(d, 1) for d in _members(case)])
    dims = _dims(case)
    if kind == "poles":
        nb = int(case["nb"])
        n, cp, ri = _pattern(dims, nb)[:3]
        return P.SelInv(n, cp, ri, perm=_order(dims, nb), dtype=P.C128, batch=int(case["poles"]))
    n, cp, ri = _pattern(dims, 1)[:3]
    return P.SelInv(n, cp, ri, perm=_order(dims, 1), batch=int(case.get("batch", 1)),
                    relax=int(case.get("relax", P.RELAX_AMALG)), unsym=1 if kind == "unsym" else 0)


def _panel_positions(h, cp, ri):
    """Positions in the X panels of the stored entries of A, from the handle's symbolic view."""
    sym = h.symbolic()
    n = int(sym["n"])
    inv = np.empty(n, np.int64)
    inv[sym["perm"]] = np.arange(n)
    r, c = inv[ri], inv[np.repeat(np.arange(n), np.diff(cp))]
    hi, lo = np.maximum(r, c), np.minimum(r, c)
    st, rp, rows, off = sym["sn_start"], sym["rowptr"], sym["rows"], sym["panel_off"]
    k = np.searchsorted(st, lo, side="right") - 1
    s, below = st[k + 1] - st[k], rp[k + 1] - rp[k]
    owner = np.repeat(np.arange(len(rp) - 1), np.diff(rp))
    at = np.searchsorted(owner * n + rows, k * n + hi) - rp[k]
    pos = np.where(hi < st[k + 1], hi - st[k], s + at)
    return off[k] + (lo - st[k]) * (s + below) + pos


def prepare(case, seed):
    kind = case["kind"]
    dev = lambda a: torch.as_tensor(a).cuda().contiguous()  # noqa: E731
    if kind == "blocks":
        L, d = _dense_blocks(case, seed)
        return dict(kind=kind, L=dev(L.transpose(1, 2).contiguous()), d=dev(d.contiguous()))
    h = _handle(case)
    st = dict(kind=kind, h=h, mode=int(case.get("mode", P.LEVEL)))
    if kind == "poles":
        blocks, z, w = _hamiltonian(case, seed)
        st.update(vals=dev(_pole_values(case, blocks, z)), w=w)
        return st
    pieces = _pieces(case, seed)
    cat = np.concatenate if kind == "uneven" else np.stack
    st["vals"] = dev(cat([_grid_values(d, diag, lo) for d, diag, lo, _ in pieces]))
    if kind == "unsym":
        st["up"] = dev(cat([_grid_values(d, diag, up) for d, diag, _, up in pieces]))
    if kind == "adjoint":
        _, cp, ri = _pattern(_dims(case), 1)[:3]
        st["pos"] = dev(_panel_positions(h, cp, ri))
        st["w"] = dev(np.random.default_rng(seed + 10 ** 6).normal(0.0, 1.0, len(ri)))
    return st


def run(state):
    kind = state["kind"]
    if kind == "blocks":
        return {"inverse": P.block_inverse_static(state["L"], state["d"])}
    h, v = state["h"], state["vals"]
    if kind == "logdet":
        theta = v.detach().requires_grad_(True)
        ld = P.logdet(theta, h)
        ld.sum().backward()
        return {"logdet": ld.detach(), "grad": theta.grad}
    if kind == "adjoint":
        theta = v.detach().requires_grad_(True)
        x = P.selected_inverse(theta, h)
        (x.index_select(1, state["pos"]) * state["w"]).sum().backward()
        return {"panels": x.detach(), "grad": theta.grad}
    if kind == "poles":
        h.factor(v)
        gamma = h.selinv_pole_sum(state["w"])
        return {"gamma": gamma, "selected": h.selected()}
    if kind == "unsym":
        h.factor_unsym(v, state["up"])
        h.selinv(state["mode"])
        return {"lower": h.selected(), "upper": h.selected_upper()}
    if kind == "indefinite":
        h.factor_bk(v)
    else:
        h.factor(v)
    h.selinv(state["mode"])
    return {"selected": h.selected()}


# --------------------------------------------------------------------------
# what a pass cannot do without, and its results in 64 bits
# --------------------------------------------------------------------------


@functools.lru_cache(maxsize=256)
def _work(key):
    case = dict(key)
    kind = case["kind"]
    if kind == "blocks":
        s, c = int(case["order"]), int(case["count"])
        return {"bytes": 8.0 * c * (s * (s + 1) / 2 + s * s), "flops": c * (s ** 3 / 3.0 + s ** 3 / 3.0)}
    h = _handle(case)
    info, sym = h.info, h.symbolic()
    s = np.diff(sym["sn_start"]).astype(np.float64)
    r = np.diff(sym["rowptr"]).astype(np.float64)
    # factorisation: diagonal blocks, panel solves and the lower triangle of the Schur update
    fac = float((s ** 3 / 3 + r * s * s + r * (r + 1) * s).sum())
    # selected inversion: steps 1-3, step 3 symmetric (non-symmetric: steps 1-4 of both triangles)
    inv = float((2 * r * r * s + 2 * r * s * s + 2 / 3 * s ** 3).sum())
    sides, es, per = 1, 8.0, 1.0
    if kind == "unsym":
        fac, inv, sides = 2 * fac, float((4 * r * r * s + 4 * r * s * s + 4 / 3 * s ** 3).sum()), 2
    if kind == "poles":
        es, per = 16.0, 4.0
    batch = float(case.get("batch", case.get("poles", 1)))
    adj = float((6 * r * r * s + 8 * r * s * s + 6 * s ** 3).sum()) if kind == "adjoint" else 0.0
    # values in, selected entries (and panels or the pole sum) out
    io = es * batch * info["nnz_a"] * 2 * sides
    if kind == "adjoint":
        io += es * info["panel_entries"] * 2 + es * 2 * info["nnz_a"]
    if kind == "poles":
        io += es * info["panel_entries"]
    h.close()
    return {"bytes": io, "flops": per * batch * (fac + inv + adj)}


def work(case):
    return dict(_work(tuple(sorted((k, v) for k, v in case.items() if k != "name"))))


def _layers(dims, nb, slot):
    """A block tridiagonal matrix by layers along the last long axis: [(A_i, lower B_i, upper B_i)] dense on
    the GPU, from slot(e, k, transposed) values [element, slot, row, column] of both triangles."""
    lower, upper = slot
    mx, my, mz = dims
    per, n = (mx * my, mz) if mz > 1 else (mx, my)  # elements of a layer, layers
    cross = 3 if mz > 1 else 2                       # the slot that leaves the layer
    _, _, _, nbr, have, _ = _pattern(dims, 1)
    out = []
    for i in range(n):
        e0 = i * per
        A = torch.zeros(per, nb, per, nb, dtype=lower.dtype, device="cuda")
        idx = torch.arange(per, device="cuda")
        A[idx, :, idx, :] = lower[e0:e0 + per, 0]
        for k in range(1, cross):
            m = torch.as_tensor(have[e0:e0 + per, k]).cuda()
            a, b = idx[m], torch.as_tensor(nbr[e0:e0 + per, k]).cuda()[m] - e0
            A[b, :, a, :] = lower[e0:e0 + per, k][m]
            A[a, :, b, :] = upper[e0:e0 + per, k][m]
        Bl = Bu = None
        if i + 1 < n:
            Bl, Bu = lower[e0:e0 + per, cross], upper[e0:e0 + per, cross]
        out.append((A.reshape(per * nb, per * nb), Bl, Bu))
    return out, per, cross, nbr, have


def _left(B, M, nb):
    """blockdiag(B) M."""
    if nb == 1:
        return B[:, 0] * M
    return torch.bmm(B, M.reshape(B.shape[0], nb, -1)).reshape(M.shape)


def _right(M, B, nb):
    """M blockdiag(B)."""
    if nb == 1:
        return M * B[:, 0, 0]
    return torch.bmm(M.reshape(M.shape[0], B.shape[0], nb).transpose(0, 1), B).transpose(0, 1).reshape(M.shape)


def _selected(dims, nb, lower, upper):
    """(lower, upper) entries [element, slot, row, column] of the inverse at the positions of the pattern, and
    log|det|: block elimination layer by layer and its backward recurrence, dense in 64 bits."""
    layers, per, cross, nbr, have = _layers(dims, nb, (lower, upper))
    n = len(layers)
    inv, logdet = [], 0.0
    for i, (A, _, _) in enumerate(layers):
        if i:
            Bl, Bu = layers[i - 1][1], layers[i - 1][2]
            A = A - _right(_left(Bl, inv[i - 1], nb), Bu, nb)
        logdet = logdet + torch.linalg.slogdet(A)[1]
        inv.append(torch.linalg.inv(A))
    lo, up = torch.zeros_like(lower), torch.zeros_like(upper)
    idx = torch.arange(per, device="cuda")
    X = None
    for i in reversed(range(n)):
        S, e0 = inv[i], i * per
        if i + 1 < n:
            Bl, Bu = layers[i][1], layers[i][2]
            down = -_left_mm(X, Bl, S, nb)        # X_{i+1,i} = -X_{i+1} Bl S_i^{-1}
            SB = _right(S, Bu, nb)                # S_i^{-1} Bu
            D = down.reshape(per, nb, per, nb)
            lo[e0:e0 + per, cross] = D[idx, :, idx, :]
            U = -(SB @ X).reshape(per, nb, per, nb)
            up[e0:e0 + per, cross] = U[idx, :, idx, :]
            X = S - SB @ down
        else:
            X = S
        Y = X.reshape(per, nb, per, nb)
        lo[e0:e0 + per, 0] = up[e0:e0 + per, 0] = Y[idx, :, idx, :]
        for k in range(1, cross):
            m = torch.as_tensor(have[e0:e0 + per, k]).cuda()
            a, b = idx[m], torch.as_tensor(nbr[e0:e0 + per, k]).cuda()[m] - e0
            lo[e0 + a, k] = Y[b, :, a, :]
            up[e0 + a, k] = Y[a, :, b, :]
    return lo, up, logdet


def _left_mm(X, Bl, S, nb):
    return X @ _left(Bl, S, nb)


def _grid_slots(dims, diag, off):
    return torch.as_tensor(np.concatenate([diag[:, None], off], 1)).cuda()[:, :, None, None]


def _stored(dims, nb, blocks):
    """Entries in the order of the stored lower CSC."""
    keep = torch.as_tensor(_pattern(dims, nb)[5]).cuda()
    return blocks.permute(0, 3, 1, 2)[keep]


def _cost(dims, nb):
    mx, my, mz = dims
    per, n = (mx * my * nb, mz) if mz > 1 else (mx * nb, my)
    return 10.0 * n * float(per) ** 3


def exact(case, seed):
    kind = case["kind"]
    if kind == "blocks":
        L, d = (t.cuda() for t in _dense_blocks(case, seed))
        v = torch.linalg.inv(L)
        m = v.transpose(1, 2) @ (v / d[:, :, None])
        return {"inverse": m.reshape(m.shape[0], -1)}
    if kind == "poles":
        dims, nb = _dims(case), int(case["nb"])
        blocks, z, _ = _hamiltonian(case, seed)
        out = []
        for zl in z:
            b = torch.as_tensor(blocks.astype(np.complex128)).cuda()
            b[:, 0] -= zl * torch.eye(nb, dtype=b.dtype, device="cuda")
            t = b.transpose(2, 3).contiguous()
            out.append(_stored(dims, nb, _selected(dims, nb, b, t)[0]))
        return {"gamma": None, "selected": torch.stack(out)}
    pieces = _pieces(case, seed)
    if sum(_cost(p[0], 1) for p in pieces) > 1.5e13:
        return None
    if kind == "adjoint":
        dims, diag, off, _ = pieces[0]
        n, cp, ri = _pattern(dims, 1)[:3]
        rows = torch.as_tensor(ri.astype(np.int64)).cuda()
        cols = torch.as_tensor(np.repeat(np.arange(n), np.diff(cp))).cuda()
        A = torch.zeros(n, n, dtype=torch.float64, device="cuda")
        A[rows, cols] = A[cols, rows] = torch.as_tensor(_grid_values(dims, diag, off)).cuda()
        X = torch.linalg.inv(A)
        w = torch.as_tensor(np.random.default_rng(seed + 10 ** 6).normal(0.0, 1.0, len(ri))).cuda()
        G = A.zero_()
        G[rows, cols] = 0.5 * w
        G = G + G.T
        Q = X @ G @ X
        return {"panels": None, "grad": (-Q[rows, cols] * torch.where(rows == cols, 1.0, 2.0))[None]}
    los, ups, lds = [], [], []
    for dims, diag, lo, up in pieces:
        x, y, ld = _selected(dims, 1, _grid_slots(dims, diag, lo), _grid_slots(dims, diag, up))
        los.append(_stored(dims, 1, x))
        ups.append(_stored(dims, 1, y))
        lds.append(ld)
    if kind == "logdet":
        _, cp, ri = _pattern(pieces[0][0], 1)[:3]
        twice = torch.full((len(ri),), 2.0, dtype=torch.float64, device="cuda")
        twice[torch.as_tensor(cp[:-1]).cuda()] = 1.0
        return {"logdet": torch.stack(lds), "grad": (los[0] * twice)[None]}
    if kind == "unsym":
        return {"lower": torch.stack(los), "upper": torch.stack(ups)}
    if kind == "uneven":
        return {"selected": torch.cat(los)[None]}
    return {"selected": torch.stack(los)}
