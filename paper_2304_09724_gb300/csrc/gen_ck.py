"""Writes the Cauchy-Kovalevskaya (Lax-Wendroff) procedure of Eq. (2.6) and Section 3.1 as
straight-line CUDA in block fixed point (see fixed.cuh): 1D and 2D Burgers and 1D Euler for one
thread, 2D Euler for two lanes; and 1D and 2D Euler in FP64.

Method.  At an interface quadrature point the solution is a truncated power series in
(X, Y, t), X = (x - x_p)/dx and Y = (y - y_p)/dy, with normalised coefficients
a[m][n][k] = d^{m+n+k}W/(dX^m dY^n dt^k) / (m! n! k!), m + n + k <= 4.  The spatial slice k = 0
comes in (the upwinded reconstruction); the PDE W_t = -F(W)_x - G(W)_y gives slice k+1 from the
flux series at slice k:
    a[m][n][k+1] = -((m+1)/dx F[m+1][n][k] + (n+1)/dy G[m][n+1][k]) / (k+1).
The flux series come from Cauchy products and quotients of the state series (Euler: u = m/rho,
v = n/rho, mu = m u, mv = m v, nv = n v, p = (g-1)(E - (mu+nv)/2), H = E + p, uH, vH).
Run:  python gen_ck.py   (output is committed).
"""
import os


class GenFixed:
    """The recursion for one thread: every coefficient an Fx (two 32-bit limbs) in registers, sums of
    products in two 64-bit accumulators, the constants (1/rho0, gamma - 1, 1/3) as Fx operands.
    Walks the dependencies backwards from the outputs a[0][0][k], k = 1..4, and emits each needed
    coefficient once, so nothing outside the triangle the outputs depend on is computed."""

    def __init__(self, dim, eq):
        self.dim, self.eq = dim, eq
        self.lines = []
        self.done = {}
        self.ncomp = 1 if eq == "burgers" else (3 if dim == 1 else 4)

    def idx_ok(self, m, n, k):
        return m >= 0 and n >= 0 and k >= 0 and m + n + k <= 4 and (self.dim == 2 or n == 0)

    def state_names(self):
        if self.eq == "burgers":
            return ["w0"]
        return ["w0", "w1", "w2"] if self.dim == 1 else ["w0", "w1", "w2", "w3"]

    def sub_indices(self, m, n, k):
        for p in range(m + 1):
            for q in range(n + 1):
                for t in range(k + 1):
                    yield p, q, t

    def fx(self, name, m, n, k):
        """C name of coefficient (m,n,k) of series `name` as an Fx; emits code on first use."""
        if not self.idx_ok(m, n, k):
            return None
        key = ("fx", name, m, n, k)
        if key in self.done:
            return self.done[key]
        v = f"{name}_{m}{n}{k}"
        W = self.state_names()
        if name in W and k == 0:
            v = f"w[{W.index(name)}][{m * 5 + n}]"
        elif name in W:
            q = W.index(name)
            z = f"{m + 1} * {self.zf(f'F{q}', m + 1, n, k - 1)}"
            if self.dim == 2:
                z += f" + {n + 1} * {self.zf(f'G{q}', m, n + 1, k - 1)}"
            self.lines.append(f"  const Fx {v} = fx_split_any(fx_time<{k}>({z}, K.third) + FX_HALF, r);")
        elif name in ("u", "v"):
            num, den = W[1 if name == "u" else 2], W[0]
            acc = [f"fx_mac_int(s, {self.fx(num, m, n, k)}, -(1 << 30));"]
            for p, q, t in self.sub_indices(m, n, k):
                if (p, q, t) != (0, 0, 0):
                    acc.append(f"fx_mac(s, {self.fx(den, p, q, t)}, {self.fx(name, m - p, n - q, k - t)});")
            self.block(v + "n", acc, lead=(m, n, k) == (0, 0, 0))  # rho0 times minus the coefficient
            self.block(v, [f"fx_mac(s, {v}n, ninv);"], const=True, lead=(m, n, k) == (0, 0, 0))
        elif name == "H":
            self.lines.append(f"  const Fx {v} = fx_split({self.z(W[-1], m, n, k)} + {self.z('p', m, n, k)} + FX_HALF, {self.rng(m, n, k)});")
        else:
            raise KeyError(name)
        self.done[key] = v
        return v

    def block(self, v, acc, const=False, lead=False):
        q, r = ("<FX_C>", "r0" if lead else "r") if const else ("", "r0" if lead else "r")
        self.lines.append(f"  Fx {v}; {{ FxAcc s = fx_zero{q}(true); " + " ".join(acc)
                          + f" {v} = fx_split(fx_sum{q}(s), {r}); }}")

    @staticmethod
    def rng(m, n, k):
        return "r0" if m + n + k == 0 else "r"

    def products(self, A, B, m, n, k):
        return [f"fx_mac(s, {self.fx(A, p, q, t)}, {self.fx(B, m - p, n - q, k - t)});"
                for p, q, t in self.sub_indices(m, n, k)]

    def zf(self, name, m, n, k):
        """A flux coefficient as a 64-bit integer expression."""
        W = self.state_names()
        if self.eq == "burgers":  # u^2 / 2
            return self.half_square(m, n, k)
        one = {"F0": (W[1],), "F1": ("mu", "p"), "F2": ("uH",)} if self.dim == 1 else \
            {"F0": (W[1],), "F1": ("mu", "p"), "F2": ("mv",), "F3": ("uH",), "G0": (W[2],), "G1": ("mv",), "G2": ("nv", "p"), "G3": ("vH",)}
        return "(" + " + ".join(self.z(t, m, n, k) for t in one[name]) + ")"

    def half_square(self, m, n, k):
        """Coefficient of u^2 / 2: each unordered pair once, half of the middle square."""
        key = ("hs", m, n, k)
        if key not in self.done:
            ps = sorted({tuple(sorted(((p, q, t), (m - p, n - q, k - t)))) for p, q, t in self.sub_indices(m, n, k)})
            acc = [f"fx_mac(s, {self.fx('w0', *a)}, {self.fx('w0', *b)});" for a, b in ps if a != b]
            mid = [f"{{ FxAcc s = fx_zero(); fx_mac(s, {self.fx('w0', *a)}, {self.fx('w0', *a)}); f += fx_sum(s) >> 1; }}" for a, b in ps if a == b]
            v = f"f_{m}{n}{k}"
            self.lines.append(f"  int64_t {v}; {{ FxAcc s = fx_zero(); " + " ".join(acc) + f" {v} = fx_sum(s); }}" + " ".join(x.replace("f +=", v + " +=") for x in mid))
            self.done[key] = v
        return self.done[key]

    def z(self, name, m, n, k):
        """C name of a coefficient as a 64-bit integer."""
        key = ("z", name, m, n, k)
        if key in self.done:
            return self.done[key]
        v = f"z_{name}_{m}{n}{k}"
        W = self.state_names()
        if name in W:
            self.lines.append(f"  const int64_t {v} = fx_join({self.fx(name, m, n, k)});")
        elif name == "p":
            kin = self.z("mu", m, n, k) + (f" + {self.z('nv', m, n, k)}" if self.dim == 2 else "")
            self.lines.append(f"  const Fx e_{m}{n}{k} = fx_split({self.z(W[-1], m, n, k)} - (({kin}) >> 1) + FX_HALF, {self.rng(m, n, k)});")
            self.lines.append(f"  int64_t {v}; {{ FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_{m}{n}{k}, K.gm1); {v} = fx_sum<FX_C>(s); }}")
        else:
            A, B = {"mu": (W[1], "u"), "mv": (W[1], "v"), "nv": (W[-2], "v"), "uH": ("u", "H"), "vH": ("v", "H")}[name]
            acc = self.products(A, B, m, n, k)
            self.lines.append(f"  int64_t {v}; {{ FxAcc s = fx_zero(); " + " ".join(acc) + f" {v} = fx_sum(s); }}")
        self.done[key] = v
        return v

    def emit(self, fname):
        W = self.state_names()
        outs = []
        for q in range(self.ncomp):
            for k in range(1, 5):
                outs.append(f"  t[{q}][{k}] = fx_join({self.fx(W[q], 0, 0, k)});")
        nc = self.ncomp
        head = [
            f"// {fname}: {self.dim}D {self.eq} in block fixed point; inputs w[q][m*5+n], outputs t[q][k], k = 1..4, in",
            "// the fields' units (fixed.cuh, ck_fixed.cuh); ninv = -1/rho0 in fixed point (Euler).",
            f"FX_FN void {fname}(const Fx (&w)[{nc}][25], Fx ninv, const CkFixedConst& K, int64_t (&t)[{nc}][5], FxRange& r) {{",
            "  (void)ninv;",
        ]
        if any(", r0)" in x for x in self.lines):
            head.append("  FxRange r0{0};  // leading coefficients are in range by their scales")
        return "\n".join(head + self.lines + outs + ["}"])


class Gen:
    """The Euler recursion in FP64, for the points whose coefficients block fixed point would hold worse: the
    same walk as GenFixed, every coefficient a double."""

    def __init__(self, dim, eq):
        self.dim, self.eq = dim, eq
        self.lines = []
        self.done = {}
        self.ncomp = 3 if dim == 1 else 4

    def idx_ok(self, m, n, k):
        return m >= 0 and n >= 0 and k >= 0 and m + n + k <= 4 and (self.dim == 2 or n == 0)

    def var(self, name, m, n, k):
        """C expression for coefficient (m,n,k) of series `name`; emits code on first use."""
        if not self.idx_ok(m, n, k):
            return None
        key = (name, m, n, k)
        if key in self.done:
            return self.done[key]
        expr = self.build(name, m, n, k)
        if expr is None:
            self.done[key] = None
            return None
        v = f"{name}_{m}{n}{k}"
        self.lines.append(f"  const double {v} = {expr};")
        self.done[key] = v
        return v

    @staticmethod
    def times(i, k, v):
        """(i / k) v"""
        return v if i == k else f"{i // k}.0 * {v}" if i % k == 0 else f"({i}.0 / {k}.0) * {v}"

    # ---- series definitions ----
    def state_names(self):
        return ["w0", "w1", "w2"] if self.dim == 1 else ["w0", "w1", "w2", "w3"]

    def build(self, name, m, n, k):
        W = self.state_names()
        if name in W:
            q = W.index(name)
            if k == 0:
                return f"a[{q}][{m * 5 + n}]"
            F = self.var(f"F{q}", m + 1, n, k - 1)
            G = self.var(f"G{q}", m, n + 1, k - 1) if self.dim == 2 else None
            terms = []
            if F is not None:
                terms.append(self.times(m + 1, k, F))
            if G is not None:
                terms.append(self.times(n + 1, k, G))
            if not terms:
                return None
            return "-(" + " + ".join(terms) + ")"
        if self.dim == 1:
            r, mx, E = W
            if name == "u":
                return self.quotient(mx, r, "u", m, n, k)
            if name == "mu":
                return self.product(mx, "u", m, n, k)
            if name == "p":
                e = self.var(E, m, n, k)
                mu = self.var("mu", m, n, k)
                return f"gm1 * ({e} - 0.5 * {mu})"
            if name == "H":
                return f"{self.var(E, m, n, k)} + {self.var('p', m, n, k)}"
            if name == "uH":
                return self.product("u", "H", m, n, k)
            if name == "F0":
                return self.var(mx, m, n, k)
            if name == "F1":
                return f"{self.var('mu', m, n, k)} + {self.var('p', m, n, k)}"
            if name == "F2":
                return self.var("uH", m, n, k)
            raise KeyError(name)
        r, mx, my, E = W
        if name == "u":
            return self.quotient(mx, r, "u", m, n, k)
        if name == "v":
            return self.quotient(my, r, "v", m, n, k)
        if name == "mu":
            return self.product(mx, "u", m, n, k)
        if name == "mv":
            return self.product(mx, "v", m, n, k)
        if name == "nv":
            return self.product(my, "v", m, n, k)
        if name == "p":
            return f"gm1 * ({self.var(E, m, n, k)} - 0.5 * ({self.var('mu', m, n, k)} + {self.var('nv', m, n, k)}))"
        if name == "H":
            return f"{self.var(E, m, n, k)} + {self.var('p', m, n, k)}"
        if name == "uH":
            return self.product("u", "H", m, n, k)
        if name == "vH":
            return self.product("v", "H", m, n, k)
        if name == "F0":
            return self.var(mx, m, n, k)
        if name == "F1":
            return f"{self.var('mu', m, n, k)} + {self.var('p', m, n, k)}"
        if name == "F2":
            return self.var("mv", m, n, k)
        if name == "F3":
            return self.var("uH", m, n, k)
        if name == "G0":
            return self.var(my, m, n, k)
        if name == "G1":
            return self.var("mv", m, n, k)
        if name == "G2":
            return f"{self.var('nv', m, n, k)} + {self.var('p', m, n, k)}"
        if name == "G3":
            return self.var("vH", m, n, k)
        raise KeyError(name)

    def sub_indices(self, m, n, k):
        for p in range(m + 1):
            for q in range(n + 1):
                for t in range(k + 1):
                    yield p, q, t

    def product(self, A, B, m, n, k):
        terms = []
        for p, q, t in self.sub_indices(m, n, k):
            a = self.var(A, p, q, t)
            b = self.var(B, m - p, n - q, k - t)
            if a is not None and b is not None:
                terms.append(f"{a} * {b}")
        if not terms:
            return None
        return " + ".join(terms)

    def quotient(self, A, B, name, m, n, k):
        """name = A / B; name[g] = (A[g] - sum_{0 < b <= g} B[b] name[g - b]) / B[0], the sum
        subtracted term by term."""
        a = self.var(A, m, n, k)
        terms = []
        for p, q, t in self.sub_indices(m, n, k):
            if (p, q, t) == (0, 0, 0):
                continue
            b = self.var(B, p, q, t)
            c = self.var(name, m - p, n - q, k - t)
            if b is not None and c is not None:
                terms.append(f"{b} * {c}")
        num = a if a is not None else "0.0"
        if terms:
            # a - t1 - t2 - ... left to right: every step contracts to one fused multiply-add
            num = "(" + num + "".join(f" - {t}" for t in terms) + ")"
        return f"{num} * inv_r0"

    def emit(self, fname):
        W = self.state_names()
        outs = []
        for q in range(self.ncomp):
            for k in range(1, 5):
                outs.append(f"  tc[{q}][{k}] = {self.var(W[q], 0, 0, k)};")
        nc = self.ncomp
        head = [
            f"// {fname}: {self.dim}D Euler in FP64; inputs a[q][m*5+n] and outputs tc[q][k], k = 1..4, in units of L.",
            f"FX_FN void {fname}(const double (&a)[{nc}][25], double (&tc)[{nc}][5], double gm1) {{",
            "  const double inv_r0 = 1.0 / a[0][0];",
        ]
        return "\n".join(head + self.lines + outs + ["}"])


def flops_euler2d():
    """Floating-point operations of the 2D Euler recursion in its minimal form (a fused multiply-add
    counts 2): only the coefficients the outputs depend on, each product and quotient once."""
    idx = [(m, n, k) for k in range(4) for m in range(5 - k) for n in range(5 - k - m)]
    pairs = lambda s: sum((m + 1) * (n + 1) * (k + 1) for m, n, k in s)
    inner = [i for i in idx if i[0] + i[1] > 0]
    along = [i for i in idx if i[0] > 0]  # x-fluxes; as many y-fluxes
    total = 2 * (2 * (pairs(idx) - len(idx)) + len(idx))      # u, v
    total += 2 * (2 * pairs(idx) - len(idx))                  # mu, nv
    total += 2 * pairs(inner) - len(inner)                    # mv
    total += 2 * (2 * pairs(along) - len(along))              # uH, vH
    total += 4 * len(idx) + 2 * len(along)                    # p, H; mu + p, nv + p
    return total + 4 * 4 * sum((5 - k) * (4 - k) // 2 for k in range(4))  # time update of four fields


class GenLane:
    """2D Euler in block fixed point with two lanes per point: lane "x" carries u and the x-fluxes,
    lane "y" (16 lanes up) v and the y-fluxes.  Both run the same code in their own coordinates:
    (i, j) = (m, n) for x and (n, m) for y, vel = u / v, mom = m / n, oth = n / m; what they share (rho,
    both momenta, H) lies in shared memory, what they exchange (the two kinetic terms of p, the flux
    derivatives) goes through shuffles."""

    def __init__(self):
        self.lines = []

    def out(self, s):
        self.lines.append("  " + s)

    def run(self):
        for c in range(4):
            self.level(c)
        return "\n".join(self.lines)

    @staticmethod
    def pairs(d):
        return [(s - j, j) for s in range(d + 1) for j in range(s + 1)]

    @staticmethod
    def subs(i, j, c):
        return [(p, q, t) for p in range(i + 1) for q in range(j + 1) for t in range(c + 1)]

    def use(self, name, i, j, t):
        """A shared series' coefficient as a local of the current block, loaded on first use."""
        v = f"{name}{i}{j}{t}"
        if v not in self.loaded:
            self.loaded.add(v)
            arg = "s, " if name == "ser" else ""
            self.out(f"const Fx {v} = S.ld{name}({arg}{t}, {i}, {j});")
        return v

    def uses(self, series, i, j, c):
        for p, q, t in self.subs(i, j, c):
            self.use(series, p, q, t)

    def level(self, c):
        D = 4 - c
        rng = lambda i, j: "r0" if i + j + c == 0 else "r"
        self.out(f"// ---- slice {c}")
        # the velocity: rho vel = mom
        for i, j in self.pairs(D):
            self.out(f"Fx vel{i}{j}{c};")
        self.out("{")
        self.loaded = set()
        ps = self.pairs(D)
        for x, (i, j) in enumerate(ps):
            for i2, j2 in ps[x:x + 2]:  # loads run one target ahead of the sums
                for p, q, t in self.subs(i2, j2, c):
                    if p + q + t:
                        self.use("rho", p, q, t)
            self.out(f"{{ FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom({c}, {i}, {j}), -(1 << 30));")
            for p, q, t in self.subs(i, j, c):
                if p + q + t:
                    self.out(f"  fx_mac(s, rho{p}{q}{t}, vel{i - p}{j - q}{c - t});")
            self.out(f"  const Fx n = fx_split_any(fx_sum(s), {rng(i, j)});")
            self.out(f"  FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel{i}{j}{c} = fx_split_any(fx_sum<FX_C>(z), {rng(i, j)}); }}")
        self.out("}")
        # mom vel, then the pressure and H
        for i, j in self.pairs(D):
            self.out(f"int64_t k{i}{j}{c};")
        self.out("{")
        self.loaded = set()
        for x, (i, j) in enumerate(ps):
            for i2, j2 in ps[x:x + 2]:
                self.uses("mom", i2, j2, c)
            self.product("mom", f"k{i}{j}{c}", i, j, c)
        self.out("}")
        for i, j in self.pairs(D):
            if i >= 1:
                self.out(f"int64_t f{i}{j}{c};")
        for i, j in self.pairs(D):
            E = f"S.ldE(0, {i}, {j})" if c == 0 else f"E{i}{j}{c}"
            self.out(f"{{ const int64_t E = {E};")
            self.out(f"  const Fx e = fx_split_any(E - ((k{i}{j}{c} + S.swap(k{j}{i}{c})) >> 1) + FX_HALF, {rng(i, j)});")
            self.out(f"  FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);")
            self.out(f"  S.stH({c}, {i}, {j}, fx_split_any(E + p + FX_HALF, {rng(i, j)}));")
            if i >= 1:
                self.out(f"  f{i}{j}{c} = k{i}{j}{c} + p;")
            self.out("}")
        # the time update: (i + 1) times the lane's fluxes, added to the other lane's
        nxt = self.pairs(D - 1)
        for q in ("rho", "mom", "E") + (("oth",) if c == 3 else ()):
            for i, j in nxt:
                self.out(f"int64_t d{q}{i}{j}{c};")
        for i, j in nxt:
            self.out(f"drho{i}{j}{c} = {i + 1} * fx_join(S.ldmom({c}, {i + 1}, {j}));")
            self.out(f"dmom{i}{j}{c} = {i + 1} * f{i + 1}{j}{c};")
        # products with the other momentum and with H: one copy of the code for both (the recursion
        # alone nearly fills the instruction cache); the first go to shared memory for the other lane
        n = c + 1
        if n < 4:
            self.out("#pragma unroll 1")
            self.out("for (int s = 0; s < 2; ++s) {")
            self.loaded = set()
            for x, (i, j) in enumerate(nxt):
                for i2, j2 in nxt[x:x + 2]:
                    self.uses("ser", i2 + 1, j2, c)
                self.out(f"int64_t z{i}{j};")
                self.product("ser", f"z{i}{j}", i + 1, j, c)
                self.out(f"dE{i}{j}{c} = {i + 1} * z{i}{j};")
            self.out("if (s == 0) {")
            for i, j in nxt:
                self.out(f"  S.stoth({n}, {i}, {j}, dE{i}{j}{c});")
            self.out("} }")
            self.out("S.sync();")
        else:
            for q, series in (("oth", "oth"), ("E", "H")):
                self.out("{")
                self.loaded = set()
                for i, j in nxt:
                    self.uses(series, i + 1, j, c)
                    self.out("int64_t z;")
                    self.product(series, "z", i + 1, j, c)
                    self.out(f"d{q}{i}{j}{c} = {i + 1} * z;")
                self.out("}")
        # each lane finishes its own momentum, lane x the density, lane y the energy
        for i, j in nxt:
            other = f"S.ldown({n}, {i}, {j})" if n < 4 else f"S.swap(doth{j}{i}{c})"
            self.out(f"{{ const int64_t own = dmom{i}{j}{c} + {other};")
            self.out(f"  const int64_t both = S.pick(drho{i}{j}{c}, dE{i}{j}{c}) + S.swap(S.pick(dE{j}{i}{c}, drho{j}{i}{c}));")
            self.out(f"  S.next({n}, {i}, {j}, fx_time<{n}>(own, third), fx_time<{n}>(both, third), {'r' if n < 4 else 'r0'}); }}")
        if n < 4:
            self.out("S.sync();")
            for i, j in nxt:
                self.out(f"const int64_t E{i}{j}{n} = S.ldE({n}, {i}, {j});")

    def product(self, series, z, i, j, c):
        self.out("{ FxAcc s = fx_zero();")
        for p, q, t in self.subs(i, j, c):
            self.out(f"  fx_mac(s, {series}{p}{q}{t}, vel{i - p}{j - q}{c - t});")
        self.out(f"  {z} = fx_sum(s); }}")


def main():
    parts = ["// Generated by gen_ck.py -- do not edit.  The Cauchy-Kovalevskaya recursions",
             "// in block fixed point (see fixed.cuh, ck_fixed.cuh and gen_ck.py for the method).",
             "#pragma once", '#include "fixed.cuh"', "", "namespace shweno {", "",
             "// Constants of the recursion: 1/3 and gamma - 1.",
             "struct CkFixedConst {", "  Fx third, gm1;", "};", "",
             "// Minus z / k: from the flux derivatives of slice k - 1 to slice k.",
             "template <int K>",
             "FX_FN int64_t fx_time(int64_t z, Fx third) {",
             "  if (K == 1) return -z;",
             "  if (K == 2) return -((z + 1) >> 1);",
             "  if (K == 4) return -((z + 2) >> 2);",
             "  FxRange r0{0};",
             "  FxAcc s = fx_zero<FX_C>();",
             "  fx_mac(s, fx_split(FX_HALF - z, r0), third);",
             "  return fx_sum<FX_C>(s);", "}", ""]
    for dim, eq in ((1, "burgers"), (2, "burgers"), (1, "euler")):
        parts += [GenFixed(dim, eq).emit(f"ck_{eq}{dim}d_fx"), ""]
    parts += ["// 2D Euler, two lanes per point: S gives the shared series and constants, ninv = -1/rho0;",
              "// S.next() takes the coefficients of the next slice.",
              "template <typename Store>",
              "FX_DEV void ck_euler2d_lane(Store& S, Fx ninv, Fx gm1, Fx third, FxRange& r) {",
              "  FxRange r0{0};  // leading coefficients are in range by their scales",
              GenLane().run(), "}", ""]
    for dim in (1, 2):
        parts += [Gen(dim, "euler").emit(f"ck_euler{dim}d"), ""]
    parts.append("}  // namespace shweno")
    out = os.path.join(os.path.dirname(os.path.abspath(__file__)), "ck_fixed_generated.cuh")
    with open(out, "w") as f:
        f.write("\n".join(parts) + "\n")


if __name__ == "__main__":
    main()
