"""The work that a user of this library has it do, as cases that can be timed.

Every case is one call (or, for a whole local update, the few calls of a window
optimisation) through the public entry points of ``paper_1501_05504_gb300.binding``
on device data:

* ``heff``       the prepared H_eff operator applied to a vector (the Lanczos loop)
* ``apply``      the one-shot H_eff application (energy evaluations)
* ``expand``     the subspace-expansion term, either direction
* ``env``        the environment recursion, either direction
* ``grad``       the MPO-entry gradient of one site (the backward direction)
* ``eig``        the local eigensolver
* ``update``     a whole local update of a fresh two-site window

on the four models of this repository's workloads: the dense Heisenberg chain
(``dense``, one block), the XXZ chain (``xxz``, U(1) blocks), the Hubbard chain
(``hubbard``, U(1) x U(1) blocks) and the S=1/2 Heisenberg model on the width-4
cylinder (``cylinder``, U(1) blocks, w = 14).  Bond sectors follow the discretised
Gaussians in the charges that the repository's seeded inputs use.

Centre tensors carry Schmidt weights that fall from 1 to 1e-5 inside every
bond; tensors entering an environment update are (nearly) isometric; environment
blocks have entries of size 1/sqrt(D), symmetric under conjugation of the channels,
with the identity in the channel where nothing has been placed yet.
"""
import itertools
import math

import numpy as np
import torch

from paper_1501_05504_gb300 import binding as b

DECAY = 1e-5          # smallest Schmidt weight of a bond, relative to the largest
ALPHA = 1e-2          # mixing factor of the expansion
KMAX = 40             # Lanczos steps of the eigensolver cases (the library's default)


# ---- models -----------------------------------------------------------------------

def _spin_mpo(reach, bonds, nsym):
    """Central MPO tensor of a spin-1/2 model whose bonds end on the current site
    at the distances ``bonds`` (all <= reach); channel 0 = finished, then (S+, S-, Sz)
    for every open distance, last = nothing placed yet."""
    up = np.array([[0.0, 1.0], [0.0, 0.0]])
    ops, conj = (up, up.T, np.diag([0.5, -0.5])), (up.T, up, np.diag([0.5, -0.5]))
    coef, one = (0.5, 0.5, 1.0), np.eye(2)
    w = 2 + 3 * reach
    W = np.zeros((2, 2, w, w))
    W[:, :, 0, 0] = W[:, :, w - 1, w - 1] = one
    for a in range(3):
        W[:, :, w - 1, 1 + a] = ops[a]
        for r in range(reach):
            if r + 1 < reach:
                W[:, :, 1 + 3 * r + a, 1 + 3 * (r + 1) + a] = one
            if r + 1 in bonds:
                W[:, :, 1 + 3 * r + a, 0] = coef[a] * conj[a]
    t = [[0]] + [[2], [-2], [0]] * reach + [[0]]
    t, qp = np.array(t), np.array([[1], [-1]])
    return (W, qp, t) if nsym else (W, qp[:, :0], t[:, :0])


def _hubbard_mpo():
    """Central MPO tensor of the Hubbard chain (t = 1, U = 8), basis 2 n_up + n_dn."""
    a, p = np.array([[0.0, 1.0], [0.0, 0.0]]), np.diag([1.0, -1.0])
    one = np.eye(2)
    cu, cd = np.kron(a, one), np.kron(p, a)
    P = np.kron(p, p)
    n = np.diag([0.0, 1.0])
    W = np.zeros((4, 4, 6, 6))
    W[:, :, 0, 0] = W[:, :, 5, 5] = np.eye(4)
    for ch, (first, second) in enumerate(((cu.T @ P, cu), (cu @ P, -cu.T), (cd.T @ P, cd), (cd @ P, -cd.T))):
        W[:, :, 5, 1 + ch] = first
        W[:, :, 1 + ch, 0] = -second
    W[:, :, 5, 0] = 8.0 * np.kron(n, n)
    qp = np.array([[0, 0], [1, -1], [1, 1], [2, 0]])
    t = np.array([[0, 0], [1, 1], [-1, -1], [1, -1], [-1, 1], [0, 0]])
    return W, qp, t


def _model(name):
    """(W, qp, t, conjugate channel of every channel)."""
    if name == "hubbard":
        return _hubbard_mpo() + ([0, 2, 1, 4, 3, 5],)
    reach, bonds = (4, (1, 4)) if name == "cylinder" else (1, (1,))
    W, qp, t = _spin_mpo(reach, bonds, name != "dense")
    pair = [0] + [1 + 3 * r + a for r in range(reach) for a in (1, 0, 2)] + [t.shape[0] - 1]
    return W, qp, t, pair


GRID = {   # sigma, step and span of the charge grid of every model's bonds
    "xxz": ((3.0,), (2,), (6,)),
    "cylinder": ((5.0,), (2,), (8,)),
    "hubbard": ((2.0, 2.0), (1, 2), (5, 4)),
}


def _bond(name, m, site):
    """(charges (nsec, nsym), dims) of bond `site` (0, 1, 2, ... from the window's left)."""
    if name == "dense":
        return np.zeros((1, 0), np.int64), np.array([m], np.int64)
    sigma, step, span = GRID[name]
    odd = (site + 1) % 2
    centre = (31 + site, odd) if name == "hubbard" else (odd,)
    axes = [c + s * np.arange(-n, n + 1) for c, s, n in zip(centre, step, span)]
    q = np.array(list(itertools.product(*axes)), np.int64)
    wt = np.exp(-0.5 * (((q - np.array(centre)) / np.array(sigma)) ** 2).sum(1))
    if name == "hubbard":     # only N + 2 S^z even exists
        ok = q.sum(1) % 2 == 0
        q, wt = q[ok], wt[ok]
    raw = wt / wt.sum() * m
    dim = np.maximum(1, np.floor(raw)).astype(np.int64)
    while dim.sum() < m:
        dim[np.argmax(raw - dim)] += 1
    while dim.sum() > m and dim.max() > 1:
        dim[np.argmax(dim)] -= 1
    return q, dim


# ---- block structure (the canonical layout of the C ABI) ------------------------------

def _at(q, v):
    hit = np.nonzero((q == v).all(1))[0]
    return int(hit[0]) if len(hit) else -1


def _site_blocks(qp, left, right):
    """[(s, i, j, offset, rows, cols)], elements."""
    out, off = [], 0
    for s in range(len(qp)):
        for i in range(len(left[1])):
            j = _at(right[0], left[0][i] + qp[s])
            if j >= 0:
                out.append((s, i, j, off, int(left[1][i]), int(right[1][j])))
                off += out[-1][4] * out[-1][5]
    return out, off


def _env_blocks(t, bond):
    """[(b, bra, ket, offset, rows, cols)], elements."""
    out, off = [], 0
    for c in range(len(t)):
        for k in range(len(bond[1])):
            i = _at(bond[0], bond[0][k] + t[c])
            if i >= 0:
                out.append((c, i, k, off, int(bond[1][i]), int(bond[1][k])))
                off += out[-1][4] * out[-1][5]
    return out, off


def _fused(bond, t):
    """The expansion's bond: (charges, dims, {(channel, sector): (sector, first state)})."""
    src = {}
    for c in range(len(t)):
        for j in range(len(bond[1])):
            src.setdefault(tuple(int(x) for x in bond[0][j] + t[c]), []).append((c, j))
    qs, dims, where = sorted(src), [], {}
    for k, q in enumerate(qs):
        n = 0
        for c, j in sorted(src[q]):
            where[(c, j)] = (k, n)
            n += int(bond[1][j])
        dims.append(n)
    return (np.array(qs, np.int64).reshape(len(qs), bond[0].shape[1]), np.array(dims, np.int64)), where


# ---- inputs -------------------------------------------------------------------------

def _weights(bond, dev):
    """Schmidt weights of a bond's states, per sector: geometric from 1 to DECAY."""
    return [DECAY ** (torch.arange(int(n), dtype=torch.float64, device=dev) / max(int(n) - 1, 1)) for n in bond[1]]


def _centre_tensor(gen, qp, left, right):
    blocks, n = _site_blocks(qp, left, right)
    x = torch.randn(max(n, 1), dtype=torch.float64, device="cuda", generator=gen)
    wl, wr = _weights(left, "cuda"), _weights(right, "cuda")
    for s, i, j, off, r, c in blocks:
        x[off:off + r * c].view(r, c).mul_(torch.sqrt(wl[i][:, None] * wr[j][None, :]))
    return x / x.norm()


def _isometry(gen, qp, left, right, dirn):
    """Entries scaled so that the columns (dirn > 0) or rows (dirn < 0) are nearly orthonormal."""
    blocks, n = _site_blocks(qp, left, right)
    x = torch.randn(max(n, 1), dtype=torch.float64, device="cuda", generator=gen)
    tot = {}
    for s, i, j, off, r, c in blocks:
        k = j if dirn > 0 else i
        tot[k] = tot.get(k, 0) + (r if dirn > 0 else c)
    for s, i, j, off, r, c in blocks:
        x[off:off + r * c].mul_(1.0 / math.sqrt(tot[j if dirn > 0 else i]))
    return x


def _environment(gen, t, bond, pair, identity):
    blocks, n = _env_blocks(t, bond)
    x = torch.randn(max(n, 1), dtype=torch.float64, device="cuda", generator=gen)
    at = {(c, i, k): (off, r, n_) for c, i, k, off, r, n_ in blocks}

    def view(key):
        off, r, n_ = at[key]
        return x[off:off + r * n_].view(r, n_)
    for c, i, k, off, r, n_ in blocks:
        v = view((c, i, k))
        if c == identity:
            v.copy_(torch.eye(r, dtype=torch.float64, device="cuda"))
        elif pair[c] < c:
            v.copy_(view((pair[c], k, i)).t())
        elif pair[c] == c and i == k:
            v.copy_((0.5 / math.sqrt(r)) * (v + v.t()))
        elif pair[c] == c and i > k:
            v.copy_(view((c, k, i)).t())
        else:
            v.mul_(1.0 / math.sqrt(max(r, n_)))
    return x


def _inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    W, qp, t, pair = _model(case["model"])
    bonds = [_bond(case["model"], case["m"], k) for k in range(3)]
    last = len(t) - 1
    p = {"W": W, "qp": qp, "t": t, "bonds": bonds}
    kind, dirn = case["kind"], case.get("dir", 1)
    right = 2 if kind == "update" else 1
    p["L"] = _environment(gen, t, bonds[0], pair, last)
    p["R"] = _environment(gen, t, bonds[right], pair, 0)
    if kind == "env":
        p["M"] = _isometry(gen, qp, bonds[0], bonds[1], dirn)
    else:
        p["M"] = _centre_tensor(gen, qp, bonds[0], bonds[1])
    if kind == "update":
        p["M1"] = _isometry(gen, qp, bonds[1], bonds[2], -1)
    return p


def _workspace(case):
    return 8 << 30 if case["model"] == "cylinder" else 1 << 30


def prepare(case, seed):
    p = _inputs(case, seed)
    B = [b.Bond(q, d) for q, d in p["bonds"]]
    kind = case["kind"]
    s = {"kind": kind, "prec": case["prec"], "dir": case.get("dir", 1), "ctx": b.dmrg3s_create(0, _workspace(case))}
    s["W"] = b.MpoSite(p["qp"], p["t"], p["t"], p["W"])
    s["L"] = b.Env(p["t"], B[0], p["L"])
    s["R"] = b.Env(p["t"], B[2] if kind == "update" else B[1], p["R"])
    s["M"] = b.Site(p["qp"], B[0], B[1], p["M"])
    if kind == "heff":
        s["out"] = b.Site(p["qp"], B[0], B[1], torch.empty_like(p["M"]))
        s["op"] = b.HeffOp(s["ctx"], s["L"], s["W"], s["R"], s["M"], s["prec"])
    elif kind == "apply":
        s["out"] = b.Site(p["qp"], B[0], B[1], torch.empty_like(p["M"]))
    elif kind == "expand":
        f = b.expanded_bond(B[1] if s["dir"] > 0 else B[0], p["t"])
        s["out"] = b.empty_site_like(p["qp"], B[0], f) if s["dir"] > 0 else b.empty_site_like(p["qp"], f, B[1])
    elif kind == "env":
        s["out"] = b.empty_env(p["t"], B[1] if s["dir"] > 0 else B[0])
    elif kind == "grad":
        s["out"] = torch.empty(p["W"].size, dtype=torch.float64, device="cuda")
    elif kind == "eig":
        s["start"] = p["M"]
        s["M"] = b.Site(p["qp"], B[0], B[1], torch.empty_like(p["M"]))
    elif kind == "update":
        s["M1"] = b.Site(p["qp"], B[1], B[2], p["M1"])
        s["opts"] = b.update_opts(case["m"], kmax=KMAX, tol=1e-14, prec=s["prec"])
    return s


def run(s):
    kind = s["kind"]
    if kind == "heff":
        s["op"].apply(s["M"], s["out"])
        return {"HA": s["out"].data}
    if kind == "apply":
        b.dmrg3s_apply_heff(s["ctx"], s["L"], s["W"], s["R"], s["M"], s["out"], s["prec"])
        return {"HA": s["out"].data}
    if kind == "expand":
        b.dmrg3s_expand(s["ctx"], s["dir"], s["L"] if s["dir"] > 0 else s["R"], s["W"], s["M"], ALPHA, s["out"], s["prec"])
        return {"P": s["out"].data}
    if kind == "env":
        b.dmrg3s_update_env(s["ctx"], s["dir"], s["L"] if s["dir"] > 0 else s["R"], s["W"], s["M"], s["out"], s["prec"])
        return {"E": s["out"].data}
    if kind == "grad":
        b.dmrg3s_mpo_grad_site(s["ctx"], s["L"], s["W"], s["R"], s["M"], s["out"])
        return {"G": s["out"]}
    if kind == "eig":     # the eigensolver overwrites its start vector
        s["M"].data.copy_(s["start"])
        lam, it = b.dmrg3s_eigensolve(s["ctx"], s["L"], s["W"], s["R"], s["M"], KMAX, 1e-14, s["prec"])
        return {"lambda": lam, "iterations": it, "M": s["M"].data}
    st = b.dmrg3s_state_create(s["ctx"], [s["W"], s["W"]], [s["M"], s["M1"]], s["L"], s["R"], 0)
    info = b.dmrg3s_local_update(st, 1, ALPHA, s["opts"])
    # the updated state by its gauge-invariant part: the MPO-entry gradients of both
    # sites (the tensors themselves are defined up to a sign per kept state)
    G, _, n2 = b.dmrg3s_mpo_grad(st, shapes=[s["W"].W.shape] * 2)
    st.close()
    return {"lambda": info["lambda"], "energy_before": info["energy_before"], "energy_after": info["energy_after"],
            "discarded": info["discarded_weight"], "iterations": info["lanczos_iters"], "bond": info["new_bond_dim"],
            "norm2": n2, "G": G}


# ---- work ---------------------------------------------------------------------------

def work(case):
    W, qp, t, _ = _model(case["model"])
    l, r = _bond(case["model"], case["m"], 0), _bond(case["model"], case["m"], 1)
    mb, nm = _site_blocks(qp, l, r)
    lb, nl = _env_blocks(t, l)
    rb, nr = _env_blocks(t, r)
    rev = case["kind"] in ("expand", "env") and case.get("dir", 1) < 0
    f1 = f2 = f3 = 0.0
    # stage 1: L M (or M R), stage 2: one multiply-add per MPO entry and element,
    # stage 3: the second environment (or the bra tensor)
    terms = {}
    for s, i, j, _, rows, cols in mb:
        for c, bra, ket, _, br_, kt_ in (rb if rev else lb):
            if ket != (j if rev else i):
                continue
            a, d = (rows, br_) if rev else (br_, cols)
            f1 += 2.0 * a * d * (cols if rev else rows)
            for so in range(len(qp)):
                for e in range(len(t)):
                    if (W[so, s, e, c] if rev else W[so, s, c, e]) != 0.0:
                        f2 += 2.0 * a * d
                        terms[(e, so, i if rev else bra, bra if rev else j)] = (a, d)
    kind = case["kind"]
    dims_l, dims_r = l[1], r[1]
    for (e, so, x, y), (a, d) in terms.items():
        if kind in ("heff", "apply", "eig", "update"):
            z = _at(r[0], r[0][y] + t[e])
            f3 += 2.0 * a * d * (dims_r[z] if z >= 0 else 0)
        elif kind == "env" and not rev:
            z = _at(r[0], l[0][x] + qp[so])
            f3 += 2.0 * a * d * (dims_r[z] if z >= 0 else 0)
        elif kind == "env":
            z = _at(l[0], r[0][y] - qp[so])
            f3 += 2.0 * a * d * (dims_l[z] if z >= 0 else 0)
    if kind in ("heff", "apply"):
        return {"flops": f1 + f2 + f3, "bytes": 8.0 * (nl + nr + 2 * nm)}
    if kind in ("eig", "update"):
        # KMAX products, two Gram-Schmidt passes against up to KMAX vectors
        return {"flops": KMAX * (f1 + f2 + f3) + 4.0 * KMAX * KMAX * nm, "bytes": 8.0 * (nl + nr + 2 * nm)}
    if kind == "expand":
        f, _ = _fused(l if rev else r, t)
        _, n = _site_blocks(qp, f, r) if rev else _site_blocks(qp, l, f)
        return {"flops": f1 + f2, "bytes": 8.0 * ((nr if rev else nl) + nm + n)}
    if kind == "env":
        return {"flops": f1 + f2 + f3, "bytes": 8.0 * (nl + nr + nm)}
    # gradient: L M, M R and one inner product per entry of the MPO tensor
    fy = sum(2.0 * rows * cols * k for s, i, j, _, rows, cols in mb for c, bra, ket, _, k, n in rb if bra == j)
    return {"flops": f1 + fy, "bytes": 8.0 * (nl + nr + nm + W.size)}


# ---- the same in 64 bits --------------------------------------------------------------

def _offsets(bond):
    return np.concatenate([[0], np.cumsum(bond[1])])


def _dense(x, blocks, n, rows, cols):
    """Dense (n, rows, cols) tensor of a flat block tensor."""
    ro, co = _offsets(rows), _offsets(cols)
    D = torch.zeros(n, int(ro[-1]), int(co[-1]), dtype=torch.float64, device="cuda")
    for a, i, j, off, r, c in blocks:
        D[a, ro[i]:ro[i + 1], co[j]:co[j + 1]] = x[off:off + r * c].view(r, c)
    return D


def _flat(D, blocks, n, rows, cols):
    ro, co = _offsets(rows), _offsets(cols)
    x = torch.zeros(max(n, 1), dtype=torch.float64, device="cuda")
    for a, i, j, off, r, c in blocks:
        x[off:off + r * c] = D[a, ro[i]:ro[i + 1], co[j]:co[j + 1]].reshape(-1)
    return x


def _left_side(W, L, A):
    """T2[br][s'] = sum W[s', s, bl, br] L[bl] A[s]."""
    w, d = W.shape[3], W.shape[0]
    T2 = [[torch.zeros_like(A[0]) for _ in range(d)] for _ in range(w)]
    for bl in range(W.shape[2]):
        for s in range(d):
            x = L[bl] @ A[s]
            for so, br in zip(*np.nonzero(W[:, s, bl, :])):
                T2[br][so].add_(x, alpha=float(W[so, s, bl, br]))
    return T2


def _right_side(W, R, A):
    """U2[bl][s'] = sum W[s', s, bl, br] A[s] R[br]^T."""
    w, d = W.shape[2], W.shape[0]
    U2 = [[torch.zeros_like(A[0]) for _ in range(d)] for _ in range(w)]
    for br in range(W.shape[3]):
        for s in range(d):
            x = A[s] @ R[br].t()
            for so, bl in zip(*np.nonzero(W[:, s, :, br])):
                U2[bl][so].add_(x, alpha=float(W[so, s, bl, br]))
    return U2


def _heff(W, L, R, A):
    T2 = _left_side(W, L, A)
    out = torch.zeros_like(A)
    for br in range(W.shape[3]):
        for so in range(W.shape[0]):
            out[so] += T2[br][so] @ R[br].t()
    return out


def _lanczos(apply, x, k):
    """Ritz pair of lowest energy after k steps (Gram-Schmidt twice against all)."""
    shape = x.shape
    V = [(x / x.norm()).reshape(-1)]
    al, be = [], []
    for n in range(k):
        w = apply(V[-1].view(shape)).reshape(-1)
        B = torch.stack(V)
        h = B @ w
        w = w - B.t() @ h
        al.append(float(h[-1]))
        w = w - B.t() @ (B @ w)
        be.append(float(w.norm()))
        V.append(w / be[-1])
    T = np.diag(al) + np.diag(be[:-1], 1) + np.diag(be[:-1], -1)
    lam, Y = np.linalg.eigh(T)
    y = Y[:, 0]
    y = y if y[np.argmax(np.abs(y))] > 0 else -y
    v = torch.stack(V[:-1]).t() @ torch.from_numpy(np.ascontiguousarray(y)).cuda()
    return float(lam[0]), (v / v.norm()).view(shape)


def exact(case, seed):
    p = _inputs(case, seed)
    W, qp, t = p["W"], p["qp"], p["t"]
    l, r = p["bonds"][0], p["bonds"][1]
    kind, dirn, d, w = case["kind"], case.get("dir", 1), len(qp), len(t)
    mb, nm = _site_blocks(qp, l, r)
    lb, nl = _env_blocks(t, l)
    rb, nr = _env_blocks(t, r)
    A = _dense(p["M"], mb, d, l, r)
    if kind in ("heff", "apply"):
        return {"HA": _flat(_heff(W, _dense(p["L"], lb, w, l, l), _dense(p["R"], rb, w, r, r), A), mb, nm, l, r)}
    if kind == "eig":
        L, R = _dense(p["L"], lb, w, l, l), _dense(p["R"], rb, w, r, r)
        lam, v = _lanczos(lambda x: _heff(W, L, R, x), A, KMAX)
        return {"lambda": lam, "iterations": None, "M": _flat(v, mb, nm, l, r)}
    if kind == "grad":
        L, R = _dense(p["L"], lb, w, l, l), _dense(p["R"], rb, w, r, r)
        G = torch.zeros(d, d, w, w, dtype=torch.float64, device="cuda")
        for br in range(w):
            for so in range(d):
                Y = A[so] @ R[br]
                for bl in range(w):
                    LY = L[bl].t() @ Y
                    for s in range(d):
                        G[so, s, bl, br] = (LY * A[s]).sum()
        return {"G": G.reshape(-1)}
    if kind == "expand":
        f, where = _fused(r if dirn > 0 else l, t)
        fo, so_, base = _offsets(f), _offsets(r if dirn > 0 else l), (r if dirn > 0 else l)
        T = _left_side(W, _dense(p["L"], lb, w, l, l), A) if dirn > 0 else _right_side(W, _dense(p["R"], rb, w, r, r), A)
        D = torch.zeros((d, A.shape[1], int(fo[-1])) if dirn > 0 else (d, int(fo[-1]), A.shape[2]), dtype=torch.float64, device="cuda")
        for (c, j), (k, first) in where.items():
            to, n = int(fo[k]) + first, int(base[1][j])
            for so in range(d):
                if dirn > 0:
                    D[so, :, to:to + n] = ALPHA * T[c][so][:, so_[j]:so_[j + 1]]
                else:
                    D[so, to:to + n, :] = ALPHA * T[c][so][so_[j]:so_[j + 1], :]
        rows, cols = (l, f) if dirn > 0 else (f, r)
        pb, n = _site_blocks(qp, rows, cols)
        return {"P": _flat(D, pb, n, rows, cols)}
    if kind == "env" and dirn > 0:
        T2 = _left_side(W, _dense(p["L"], lb, w, l, l), A)
        E = torch.stack([sum(A[so].t() @ T2[c][so] for so in range(d)) for c in range(w)])
        return {"E": _flat(E, rb, nr, r, r)}
    if kind == "env":
        U2 = _right_side(W, _dense(p["R"], rb, w, r, r), A)
        E = torch.stack([sum(A[so] @ U2[c][so].t() for so in range(d)) for c in range(w)])
        return {"E": _flat(E, lb, nl, l, l)}
    return None     # a whole update: the SVD of an expansion has no short plain form


# ---- the cases ------------------------------------------------------------------------

def listed():
    return [
        # the smallest products: the dense L = 20 Heisenberg chain, one block per tensor
        {"name": "heff_dense_m64", "kind": "heff", "model": "dense", "m": 64, "prec": "fp64"},
        # a Lanczos product at the centre of the XXZ chain: FP64 (final sweeps) and 3xTF32 (bulk sweeps)
        {"name": "heff_xxz_m512", "kind": "heff", "model": "xxz", "m": 512, "prec": "fp64"},
        {"name": "heff_xxz_m512_tf32x3", "kind": "heff", "model": "xxz", "m": 512, "prec": "tf32x3"},
        # the energy after a truncation on the Hubbard chain: many small blocks, one call
        {"name": "apply_hubbard_m1024", "kind": "apply", "model": "hubbard", "m": 1024, "prec": "fp64"},
        # the largest contraction: a bulk-precision Lanczos product on the cylinder
        {"name": "heff_cylinder_m2048_tf32x3", "kind": "heff", "model": "cylinder", "m": 2048, "prec": "tf32x3"},
        # the expansion term of a right-to-left update on the Hubbard chain
        {"name": "expand_hubbard_m1024_rl", "kind": "expand", "model": "hubbard", "m": 1024, "dir": -1, "prec": "fp64"},
        # the environment of a left-to-right update on a chain whose bond is still growing
        {"name": "env_xxz_m389_lr", "kind": "env", "model": "xxz", "m": 389, "dir": 1, "prec": "fp64"},
        # the environment of a right-to-left update at the cylinder's full size
        {"name": "env_cylinder_m2048_rl", "kind": "env", "model": "cylinder", "m": 2048, "dir": -1, "prec": "fp64"},
        # the coupling derivatives: one site's MPO-entry gradient
        {"name": "grad_hubbard_m512", "kind": "grad", "model": "hubbard", "m": 512, "prec": "fp64"},
        # local eigenproblems of the two precisions of a sweep's ladder
        {"name": "eig_xxz_m512_tf32x3", "kind": "eig", "model": "xxz", "m": 512, "prec": "tf32x3"},
        {"name": "eig_xxz_m512", "kind": "eig", "model": "xxz", "m": 512, "prec": "fp64"},
        # a whole FP64 local update (eigensolver, expansion, truncation, environment, energy)
        # of a fresh window, and the gradients of the updated state
        {"name": "update_xxz_m512", "kind": "update", "model": "xxz", "m": 512, "prec": "fp64"},
    ]


RANGE = {"dense": (16, 128), "xxz": (64, 512), "hubbard": (128, 1024), "cylinder": (256, 2048)}


def draw(rng):
    kind = rng.choice(("heff", "heff", "apply", "expand", "env", "grad", "eig", "update"))
    models = ("xxz",) if kind in ("eig", "update") else ("dense", "xxz", "hubbard", "cylinder")
    model = rng.choice(models)
    lo, hi = RANGE[model]
    if kind == "update":
        lo = 256
    c = {"kind": kind, "model": model, "m": int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))}
    if kind in ("expand", "env"):
        c["dir"] = rng.choice((1, -1))
    # the library runs FP64 throughout; the products of H_eff also run in 3xTF32
    c["prec"] = rng.choice(("fp64", "tf32x3")) if kind in ("heff", "eig") else "fp64"
    return c
