"""The IP-DG Poisson system in extended precision (np.longdouble), from its
definition, for meshes on which an FP64 reference is too coarse (its Jacobians
lose the ratio of position to thickness). Cell-local DOFs, nodes x-fastest."""
import numpy as np

LD = np.longdouble


def gauss(n):
    s = np.sqrt
    if n == 2:
        x, w = [-s(LD(1) / 3), s(LD(1) / 3)], [1, 1]
    elif n == 3:
        x, w = [-s(LD(3) / 5), 0, s(LD(3) / 5)], [LD(5) / 9, LD(8) / 9, LD(5) / 9]
    else:
        a, b = s(LD(3) / 7 - LD(2) / 7 * s(LD(6) / 5)), s(LD(3) / 7 + LD(2) / 7 * s(LD(6) / 5))
        u, v = (18 + s(LD(30))) / 36, (18 - s(LD(30))) / 36
        x, w = [-b, -a, a, b], [v, u, u, v]
    return (np.array(x, dtype=LD) + 1) / 2, np.array(w, dtype=LD) / 2


def lagrange(p, x):
    """Values and derivatives of the polynomials on the nodes m / p at x: [..., p + 1]."""
    x = np.asarray(x, dtype=LD)
    v, d = [], []
    for m in range(p + 1):
        val, der = np.ones_like(x), np.zeros_like(x)
        for s in range(p + 1):
            if s != m:
                den = LD(m - s) / p
                der = der * (x - LD(s) / p) / den + val / den
                val = val * (x - LD(s) / p) / den
        v.append(val)
        d.append(der)
    return np.stack(v, -1), np.stack(d, -1)


def shapes(p, x):
    """phi [n, nb] and its reference gradient [n, nb, 3] at points x [n, 3]."""
    V, D = zip(*(lagrange(p, x[:, k]) for k in range(3)))
    def tensor(a, b, c):
        return np.einsum("ni,nj,nk->nkji", a, b, c).reshape(x.shape[0], -1)
    g = [tensor(D[0], V[1], V[2]), tensor(V[0], D[1], V[2]), tensor(V[0], V[1], D[2])]
    return tensor(*V), np.stack(g, -1)


def geometry(xv, x):
    """Cofactors [n, 3, 3] and determinant of the trilinear map of the vertices xv [8, 3]."""
    d = xv.astype(LD) - xv[0].astype(LD)  # differences first: exact for neighbouring positions
    J = np.einsum("ak,nad->nkd", d, shapes(1, x)[1])
    cof = np.empty_like(J)
    for k in range(3):
        for j in range(3):
            k1, k2, j1, j2 = (k + 1) % 3, (k + 2) % 3, (j + 1) % 3, (j + 2) % 3
            cof[:, k, j] = J[:, k1, j1] * J[:, k2, j2] - J[:, k1, j2] * J[:, k2, j1]
    return cof, np.einsum("nd,nd->n", J[:, 0], cof[:, 0])


def corner(f, s, t):
    ax = [k for k in range(3) if k != f // 2]
    return ((f % 2) << (f // 2)) | (s << ax[0]) | (t << ax[1])


def dg_values(mesh, p, tau, gamma, facets, row_ptr, col):
    """The CSR values (longdouble) for the pattern (row_ptr, col)."""
    nb = (p + 1) ** 3
    xv = np.asarray(mesh.coords)[mesh.cell_vertices]
    g, w = gauss(p + 1)
    pt3 = np.array([(x, y, z) for z in g for y in g for x in g])
    w3 = np.array([a * b * c for c in w for b in w for a in w])
    wst = np.array([a * b for b in w for a in w])
    st = np.array([(a, b) for b in g for a in g])
    blocks = {}

    def add(e, f, m):
        blocks[e, f] = blocks.get((e, f), 0) + m

    phi, dphi = shapes(p, pt3)
    for e in range(mesh.n_cells):
        cof, det = geometry(xv[e], pt3)
        gr = np.einsum("nkd,nad->nak", cof, dphi)
        add(e, e, np.einsum("n,nak,nbk->ab", w3 / det, gr, gr))

    def side(e, verts):
        """Reference points on cell e whose face corners (s, t) are the local vertices verts."""
        c = np.array([[(v >> k) & 1 for k in range(3)] for v in verts], dtype=LD)
        s, t = st[:, :1], st[:, 1:]
        return c[0] * (1 - s) * (1 - t) + c[1] * s * (1 - t) + c[2] * (1 - s) * t + c[3] * s * t

    plus, minus, pf, mf, bc, bf = facets
    for i in range(len(plus) + len(bc)):
        interior = i < len(plus)
        e = [plus[i], minus[i]] if interior else [bc[i - len(plus)]]
        f = pf[i] if interior else bf[i - len(plus)]
        verts = [corner(f, c & 1, c >> 1) for c in range(4)]
        local = [verts]
        if interior:
            ids = list(mesh.cell_vertices[e[1]])
            local.append([ids.index(mesh.cell_vertices[e[0]][v]) for v in verts])
        ph, gn = [], []
        for k, cell in enumerate(e):
            x = side(cell, local[k])
            cof, det = geometry(xv[cell], x)
            if k == 0:
                nd = cof[:, :, f // 2] * (1 if f % 2 else -1)
                ln = np.sqrt((nd * nd).sum(1))
                n, ds = nd / ln[:, None], ln * wst
            v, d = shapes(p, x)
            ph.append(v)
            gn.append(np.einsum("nkd,nad,nk->na", cof, d, n) / det[:, None])
        pen, half, sg = LD(gamma) / ds.sum(), LD(1) / 2 if interior else LD(1), (1, -1)
        for a in range(len(e)):
            for b in range(len(e)):
                X = np.einsum("q,qa,qb->ab", ds, ph[a], gn[b])
                Xt = np.einsum("q,qa,qb->ab", ds, gn[a], ph[b])
                Y = np.einsum("q,qa,qb->ab", ds, ph[a], ph[b])
                add(e[a], e[b], -half * sg[a] * X - LD(tau) * half * sg[b] * Xt + pen * sg[a] * sg[b] * Y)
    val = np.zeros(len(col), dtype=LD)
    rows = np.repeat(np.arange(len(row_ptr) - 1), np.diff(row_ptr))
    for k, (r, c) in enumerate(zip(rows, col)):
        val[k] = blocks[r // nb, c // nb][r % nb, c % nb]
    return val
