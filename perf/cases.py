"""The work this library is used for, as cases that can be timed and compared: the products Y = A X of
the clover Wilson-Dirac operator, the Jacobi preconditioner in its precisions, the block updates of
an iteration, the learned preconditioner's application and training step, and whole solves.

A case is a dict of plain values.  ``prepare`` makes what a user's program holds before the call (the
context of a gauge field, the right-hand sides, output buffers), ``run`` makes the call, ``exact``
gives the same result in plain 64-bit torch written from the operator's definition, and ``work``
counts the bytes and operations that a pass cannot do without.
"""
import math

import torch

import paper_0907_3261_gb300 as wd

CSW = 1.0


def listed():
    return [
        # The smallest call: one column on 4^4 (the lattice of the first parity configuration), as a
        # test or a single-source measurement makes it.  Launches and latency are all there is.
        dict(name="apply_4_L1", kind="apply", dims="4x4x4x4", L=1, kappa=0.115),
        # A middle-sized lattice of the batched workload (12^3x24) with an odd number of columns.
        dict(name="apply_12x24_L7", kind="apply", dims="12x12x12x24", L=7, kappa=0.12),
        # The paper's lattice with its twelve spin-colour columns: the product the outer method
        # makes twice per iteration.
        dict(name="apply_16x32_L12", kind="apply", dims="16x16x16x32", L=12, kappa=0.13),
        # The largest lattice of the batched workload (32^3x64) with twelve columns.
        dict(name="apply_32x64_L12", kind="apply", dims="32x32x32x64", L=12, kappa=0.12),
        # The paper's preconditioner in its own arithmetic (FP64, j = 12), on the 8^3x16 lattice of
        # the kappa scan.
        dict(name="jacobi_fp64_8x16_L12", kind="jacobi", dims="8x8x8x16", L=12, kappa=0.13, j=12,
             precision=0),
        # FP32 sweeps as the batched solves use them, at an odd number of columns.
        dict(name="jacobi_fp32_12x24_L7", kind="jacobi", dims="12x12x12x24", L=7, kappa=0.12, j=8,
             precision=1),
        # The double-float preconditioner of the default solve on the paper's lattice.
        dict(name="jacobi_df_16x32_L12", kind="jacobi", dims="16x16x16x32", L=12, kappa=0.134, j=12,
             precision=4),
        # The direction recurrences of one iteration, U = (P - zeta V) alpha and P = R + U gamma,
        # V = W + Y gamma with its Gram product, as a driver that runs the iteration itself calls them.
        dict(name="updates_df_16x32_L12", kind="updates", dims="16x16x16x32", L=12, kappa=0.13,
             precision=1),
        # The learned preconditioner applied to a block on the paper's lattice.
        dict(name="net_16x32_L12", kind="net", dims="16x16x16x32", L=12, kappa=0.13, layers=4,
             hidden=4),
        # One training step's forward and backward pass on a training configuration (8^4, L = 12).
        dict(name="net_grad_8_L12", kind="net_grad", dims="8x8x8x8", L=12, kappa=0.13, layers=4,
             hidden=4),
        # A small whole solve in the paper's arithmetic (point sources, L = 4, j = 4 on 4^4): many
        # short launches, one host decision per iteration.
        dict(name="solve_4_L4", kind="solve", dims="4x4x4x4", L=4, kappa=0.115, j=4, precision=0,
             source="point"),
        # The whole solve on the paper's lattice in the default form (double-float sweeps and
        # direction recurrences), Z4 noise sources, L = j = 12.
        dict(name="solve_16x32_L12", kind="solve", dims="16x16x16x32", L=12, kappa=0.13, j=12,
             precision=5, source="z4"),
    ]


def _draw_dims(rng, vmin, vmax):
    """Four extents of a lattice of about v sites, v spread over the logarithm; odd ones among them."""
    v = math.exp(rng.uniform(math.log(vmin), math.log(vmax)))
    d = [max(2, round(v ** 0.25 * math.exp(rng.uniform(-0.4, 0.4)))) for _ in range(3)]
    d.append(max(2, int(v / (d[0] * d[1] * d[2]))))
    return "x".join(map(str, d))


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "jacobi", "jacobi", "jacobi", "updates", "net",
                       "net_grad", "solve"])
    L = rng.randint(1, 16)
    kappa = round(rng.uniform(0.115, 0.13), 4)
    c = dict(kind=kind, L=L, kappa=kappa)
    if kind == "apply":
        c["dims"] = _draw_dims(rng, 200, 32 ** 3 * 64 * 12 / (2 * L) if L > 6 else 32 ** 3 * 64)
    elif kind == "jacobi":
        c["dims"] = _draw_dims(rng, 200, 16 ** 3 * 32)
        c.update(j=rng.randint(2, 16), precision=rng.choice([0, 0, 1, 3, 4, 4]))
    elif kind == "updates":
        c["dims"] = _draw_dims(rng, 200, 16 ** 3 * 32)
        c["precision"] = rng.choice([0, 1])
    elif kind == "net":
        c["dims"] = _draw_dims(rng, 200, 16 ** 3 * 32)
        c.update(layers=rng.randint(2, 4), hidden=rng.choice([2, 4]))
    elif kind == "net_grad":
        c["dims"] = _draw_dims(rng, 200, 8 ** 3 * 16)
        c.update(layers=rng.randint(2, 4), hidden=rng.choice([2, 4]))
    else:
        c["dims"] = _draw_dims(rng, 1000, 16 ** 3 * 24)
        c["L"] = min(L, 12)
        c.update(j=rng.choice([4, 8, 12]), precision=rng.choice([0, 5]),
                 source=rng.choice(["z4", "z4", "point"]))
    return c


# ---------------------------------------------------------------- inputs (torch, from the seed alone)
def _device():
    return torch.device("cuda") if torch.cuda.is_available() else torch.device("cpu")


def _generator(seed, stream):
    g = torch.Generator(device=_device())
    g.manual_seed(seed * 64 + stream)
    return g


def _gaussian(shape, seed, stream):
    x = torch.randn(tuple(shape) + (2,), generator=_generator(seed, stream), device=_device(),
                    dtype=torch.float64)
    return torch.view_as_complex(x)


def _dims(case):
    return tuple(int(d) for d in case["dims"].split("x"))


def _volume(dims):
    return dims[0] * dims[1] * dims[2] * dims[3]


def _links(dims, seed):
    """U = SU3proj(1 + 0.2 G): Gram-Schmidt on rows 0 and 1, row 2 = conj(row0 x row1)."""
    m = 0.2 * _gaussian((_volume(dims), 4, 3, 3), seed, 1)
    m = m + torch.eye(3, device=m.device, dtype=m.dtype)
    a = m[..., 0, :]
    a = a / torch.linalg.vector_norm(a, dim=-1, keepdim=True)
    b = m[..., 1, :]
    b = b - (a.conj() * b).sum(-1, keepdim=True) * a
    b = b / torch.linalg.vector_norm(b, dim=-1, keepdim=True)
    return torch.stack([a, b, torch.linalg.cross(a, b).conj()], dim=-2).contiguous()


def _block(case, seed, stream):
    return _gaussian((_volume(_dims(case)), 4, 3, case["L"]), seed, stream)


def _sources(case, seed):
    V, L = _volume(_dims(case)), case["L"]
    if case["source"] == "point":
        b = torch.zeros((V, 4, 3, L), dtype=torch.complex128, device=_device())
        for i in range(L):
            b[(i // 12 + seed) % V, i % 4, (i // 4) % 3, i] = 1.0
        return b
    k = torch.randint(0, 4, (V, 4, 3, L), generator=_generator(seed, 2), device=_device())
    vals = torch.tensor([1, 1j, -1, -1j], dtype=torch.complex128, device=_device())
    return vals[k]


def _weights(case, seed):
    """The initial network: identity on the on-site blocks plus noise, values that FP32 holds."""
    ch = [1] + [case["hidden"]] * (case["layers"] - 1) + [1]
    out = []
    for i in range(case["layers"]):
        cin, cout = ch[i], ch[i + 1]
        w = 0.01 * _gaussian((9, cout, cin, 4, 4), seed, 20 + i)
        for co in range(cout):
            for ci in range(cin):
                if cin == 1 or cout == 1 or co == ci:
                    w[0, co, ci] += torch.eye(4, device=w.device) * (1.0 / cin if cout == 1 else 1.0)
        out.append(w.to(torch.complex64).to(torch.complex128))
    return out


def _coef(case, seed):
    L = case["L"]
    g = _gaussian((2 * L * L + 1,), seed, 9).cpu().numpy()
    return complex(g[0]), g[1:1 + L * L].reshape(L, L), g[1 + L * L:].reshape(L, L)


def prepare(case, seed):
    kind, dims = case["kind"], _dims(case)
    links = _links(dims, seed)
    st = dict(kind=kind, case=case, ctx=wd.wd_create(links, dims, case["kappa"], CSW))
    if kind in ("apply", "jacobi"):
        st["X"] = _block(case, seed, 3)
        st["Y"] = torch.empty_like(st["X"])
    elif kind == "updates":
        for i, name in enumerate(("P", "V", "R", "W", "U", "Y", "Rt")):
            st[name] = _block(case, seed, 10 + i)
        for name in ("U_new", "P_new", "V_new"):
            st[name] = torch.empty_like(st["P"])
        st["zeta"], st["alpha"], st["gamma"] = _coef(case, seed)
    elif kind in ("net", "net_grad"):
        st["net"] = wd.wd_net_create(case["layers"], case["hidden"],
                                     [w.cpu().numpy() for w in _weights(case, seed)])
        st["X"] = _block(case, seed, 3)
        st["Y"] = torch.empty_like(st["X"]) if kind == "net" else _block(case, seed, 4)
    else:
        st["B"] = _sources(case, seed)
        st["X"] = torch.empty_like(st["B"])
    return st


def run(state):
    case, ctx, kind = state["case"], state["ctx"], state["kind"]
    if kind == "apply":
        return wd.wd_apply(ctx, state["X"], state["Y"])
    if kind == "jacobi":
        return wd.jacobi_precond(ctx, state["X"], case["j"], state["Y"], precision=case["precision"])
    if kind == "updates":
        u = wd.bb_update_u(ctx, state["P"], state["V"], state["U_new"], state["zeta"], state["alpha"],
                           precision=case["precision"])
        rtv = wd.bb_update_pv(ctx, state["P_new"], state["V_new"], state["R"], state["W"], state["U"],
                              state["Y"], state["Rt"], state["gamma"], precision=case["precision"])
        return u, state["P_new"], state["V_new"], rtv
    if kind == "net":
        return wd.wd_net_apply(ctx, state["net"], state["X"], state["Y"])
    if kind == "net_grad":
        return wd.wd_net_loss_grad(ctx, state["net"], state["X"], state["Y"])
    state["X"].zero_()
    X, _ = wd.bbicggr_solve(ctx, state["B"], state["X"], j=case["j"], tol=1e-12,
                            precision=case["precision"])
    return X


def _iterations(case):
    """Outer iterations such a solve takes, about (hopping products grow towards the critical kappa)."""
    mvm = 260.0 * (1.0 + 1.1 * (case["kappa"] - 0.115) / 0.015)
    return max(1, round(mvm / (2 * (case["j"] + 1))))


def work(case):
    """Each block, link (18 reals) and site block (72 reals) read or written once in the type of the
    call's buffers (FP64); 1824 flop per site and column of a product with A, 1872 of a Jacobi sweep,
    528 of the first one, 8 L per entry of a product with an L x L matrix."""
    V, L, kind = _volume(_dims(case)), case["L"], case["kind"]
    block, op = 192.0 * V * L, (576.0 + 576.0) * V
    if kind == "apply":
        return {"bytes": 2 * block + op, "flops": 1824.0 * V * L}
    if kind == "jacobi":
        return {"bytes": 2 * block + op, "flops": (528.0 + 1872.0 * (case["j"] - 1)) * V * L}
    if kind == "updates":
        n = 12.0 * V * L
        return {"bytes": 10 * block, "flops": n * (8 * L + 8) + n * (24 * L + 4)}
    if kind in ("net", "net_grad"):
        ch = [1] + [case["hidden"]] * (case["layers"] - 1) + [1]
        fwd = sum(8 * ch[i] * 288.0 + 9 * ch[i] * ch[i + 1] * 384.0 for i in range(case["layers"])) * V * L
        times = 1 if kind == "net" else 3
        return {"bytes": 2 * block + 576.0 * V, "flops": times * fwd}
    k, j = _iterations(case), case["j"]
    per = 2 * 1824.0 + 2 * (528.0 + 1872.0 * (j - 1)) + 12 * (48 * L + 60)
    return {"bytes": 2 * block + op, "flops": k * per * V * L}


# ---------------------------------------------------------------- plain 64-bit statement
_PAULI = [[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]]


def _gammas(dev):
    out = []
    for k in range(4):
        g = torch.zeros((4, 4), dtype=torch.complex128, device=dev)
        if k < 3:
            s = torch.tensor(_PAULI[k], dtype=torch.complex128, device=dev)
            g[:2, 2:], g[2:, :2] = -1j * s, 1j * s
        else:
            g[:2, 2:] = g[2:, :2] = torch.eye(2, dtype=torch.complex128, device=dev)
        out.append(g)
    return out


def _shift(x, dims, mu, d):
    """x(s + d mu) for a field whose first axis is the site index (x runs fastest)."""
    y = x.reshape((dims[3], dims[2], dims[1], dims[0]) + tuple(x.shape[1:]))
    return torch.roll(y, -d, dims=3 - mu).reshape(x.shape)


class _Operator:
    def __init__(self, dims, links, kappa):
        self.dims, self.kappa = dims, kappa
        self.U = [links[:, mu].contiguous() for mu in range(4)]
        self.g = _gammas(links.device)
        self.AD = None

    def transport(self, psi, mu, d):
        """U_mu(s) psi(s + mu) for d = +1, U_mu(s - mu)^H psi(s - mu) for d = -1."""
        if d > 0:
            u, p = self.U[mu], _shift(psi, self.dims, mu, 1)
        else:
            u, p = _shift(self.U[mu], self.dims, mu, -1).mH, _shift(psi, self.dims, mu, -1)
        out = torch.empty_like(psi)
        for a in range(3):
            out[:, :, a] = u[:, a, 0, None, None] * p[:, :, 0]
            for b in (1, 2):
                out[:, :, a] += u[:, a, b, None, None] * p[:, :, b]
        return out

    def spin(self, m, psi):
        out = torch.zeros_like(psi)
        for i in range(4):
            for k in range(4):
                if m[i, k] != 0:
                    out[:, i] += complex(m[i, k]) * psi[:, k]
        return out

    def hop(self, psi):
        eye = torch.eye(4, dtype=torch.complex128)
        out = torch.zeros_like(psi)
        for mu in range(4):
            g = self.g[mu].cpu()
            out += self.spin(eye - g, self.transport(psi, mu, 1))
            out += self.spin(eye + g, self.transport(psi, mu, -1))
        return out

    def site_blocks(self):
        """A_D as 12x12 matrices per site."""
        if self.AD is None:
            U, dims = self.U, self.dims
            V, dev = U[0].shape[0], U[0].device
            AD = torch.eye(12, dtype=torch.complex128, device=dev).expand(V, 12, 12).clone()
            for mu in range(4):
                for nu in range(mu + 1, 4):
                    up = lambda x, m, d: _shift(x, dims, m, d)
                    um, un = U[mu], U[nu]
                    q = um @ up(un, mu, 1) @ up(um, nu, 1).mH @ un.mH
                    um_b, un_b = up(um, mu, -1), up(un, nu, -1)
                    q = q + un @ up(up(um, mu, -1), nu, 1).mH @ up(un, mu, -1).mH @ um_b
                    q = q + um_b.mH @ up(up(un, mu, -1), nu, -1).mH @ up(up(um, mu, -1), nu, -1) @ un_b
                    q = q + un_b.mH @ up(um, nu, -1) @ up(up(un, mu, 1), nu, -1) @ um.mH
                    F = (q - q.mH) / 8j
                    sig = 0.5j * (self.g[mu] @ self.g[nu] - self.g[nu] @ self.g[mu])
                    k = torch.einsum("ij,vab->viajb", sig, F).reshape(V, 12, 12)
                    AD -= self.kappa * CSW * k
            self.AD = AD
        return self.AD

    def blocks(self, m, psi):
        V, L = psi.shape[0], psi.shape[-1]
        v = psi.reshape(V, 12, L)
        out = torch.empty_like(v)
        step = max(1, (1 << 24) // (144 + 24 * L))
        for s in range(0, V, step):
            out[s:s + step] = torch.matmul(m[s:s + step], v[s:s + step])
        return out.reshape(psi.shape)

    def apply(self, psi):
        return self.blocks(self.site_blocks(), psi) - self.kappa * self.hop(psi)


def _exact_solve(A, B):
    """BiCGStab on all columns at once, restarted from its own result (64-bit residuals)."""
    X = torch.zeros_like(B)
    dot = lambda a, b: (a.conj() * b).sum(dim=(0, 1, 2))
    nb = dot(B, B).real.sqrt()
    for _ in range(3):
        R = B - A.apply(X)
        if float((dot(R, R).real.sqrt() / nb).max()) < 3e-15:
            break
        Rt, P = R.clone(), R.clone()
        D = torch.zeros_like(B)
        rho = dot(Rt, R)
        for _ in range(400):
            v = A.apply(P)
            al = rho / dot(Rt, v)
            S = R - al * v
            t = A.apply(S)
            om = dot(t, S) / dot(t, t)
            D += al * P + om * S
            R = S - om * t
            if float((dot(R, R).real.sqrt() / nb).max()) < 1e-15:
                break
            new = dot(Rt, R)
            P = R + (new / rho) * (al / om) * (P - om * v)
            rho = new
        X = X + D
    return X


def _net_forward(op, weights, x):
    act = [x]
    for w in weights:
        moved = [[p] + [op.transport(p, mu, 1) for mu in range(4)] +
                 [op.transport(p, mu, -1) for mu in range(4)] for p in act]
        act = [sum(torch.einsum("ij,vjal->vial", w[d, co, ci], moved[ci][d])
                   for ci in range(len(act)) for d in range(9)) for co in range(w.shape[1])]
    return act[0]


def exact(case, seed):
    kind, size = case["kind"], _volume(_dims(case)) * case["L"]
    if kind == "solve" and size * _iterations(case) * case["j"] > 20_000_000:
        return None
    if kind == "updates":
        P, V, R, W, U, Y, Rt = (_block(case, seed, 10 + i) for i in range(7))
        zeta, alpha, gamma = _coef(case, seed)
        al, ga = (torch.as_tensor(m, device=P.device) for m in (alpha, gamma))
        Vn = W + Y @ ga
        flat = lambda b: b.reshape(-1, case["L"])
        rtv = sum(flat(Rt)[i:i + 65536].mH @ flat(Vn)[i:i + 65536]
                  for i in range(0, flat(Rt).shape[0], 65536))
        return (P - zeta * V) @ al, R + U @ ga, Vn, rtv.cpu().numpy()
    op = _Operator(_dims(case), _links(_dims(case), seed), case["kappa"])
    if kind == "apply":
        return op.apply(_block(case, seed, 3))
    if kind == "jacobi":
        R = _block(case, seed, 3)
        inv = torch.linalg.inv(op.site_blocks())
        G = op.blocks(inv, R)
        for _ in range(case["j"] - 1):
            G = op.blocks(inv, R + case["kappa"] * op.hop(G))
        return G
    if kind == "net":
        if size > 200_000:
            return None
        return _net_forward(op, _weights(case, seed), _block(case, seed, 3))
    if kind == "net_grad":
        ws = [w.requires_grad_(True) for w in _weights(case, seed)]
        E = _block(case, seed, 4)
        y = _net_forward(op, ws, _block(case, seed, 3))
        n = (E.abs() ** 2).sum(dim=(0, 1, 2))
        loss = (((y - E).abs() ** 2).sum(dim=(0, 1, 2)) / n).mean()
        loss.backward()
        return float(loss.detach()), [0.5 * w.grad.cpu().numpy() for w in ws]
    return _exact_solve(op, _sources(case, seed))
