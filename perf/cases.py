"""The workloads by which this library's speed is judged.

Each case is one call that a user's program makes: a time step of the shell dynamo (the reason the library
exists), an operator apply, a preconditioned solve, a batched solve, a forward pass or a gradient of the learned
coarse correction.  Grids, box splits, solver options and network sizes are those of bench.py's shells and
workloads and of the tests, plus ragged sizes between them.

listed() gives the fixed cases, draw() more of the same ranges; prepare() builds the handles and device inputs a
program holds before the call, run() is the call, work() the traffic and arithmetic it cannot do without, and
exact() what it should return, in 64 bits, from the plain torch restatement of the discretization below.
"""
import math
import weakref

import numpy as np
import torch

from paper_2009_02171_gb300 import fv
from paper_2009_02171_gb300.inputs import uneven_boxes

PHYS = dict(E=1e-3, Ra=100.0, Pr=1.0, Pm=5.0)
RI, RO = 7.0 / 13.0, 20.0 / 13.0
PREC = {'fp64': fv.FV_PREC_FP64, 'fp32': fv.FV_PREC_FP32, 'bf16': fv.FV_PREC_BF16}
KIND = {'vtbe': fv.FV_VTBE, 'ppbe': fv.FV_PPBE}


def _boxes(Ns, Nr):
    """bench.py's fine split: boxes of at most 32 x 32 x 16 cells."""
    return dict(p1=-(-Ns // 32), p2=-(-Ns // 32), p3=-(-Nr // 16))


def listed():
    return [
        # the smallest shell of the configuration list, FP64 throughout, one box a panel: launches and latency
        dict(name='step_fp64_16', op='step', Ns=16, Nr=16, prec='fp64', p1=1, p2=1, p3=1, overlap=1, levels=1, nsteps=2,
             rtol=1e-8),
        # the headline shell of bench.py in mixed precision, first step and a step with history; residuals to 1e-11 (one
        # outer iteration more than 1e-8 takes), since the pressure's relative error is about a thousand times as large
        dict(name='step_fp32_64', op='step', Ns=64, Nr=64, prec='fp32', p1=2, p2=2, p3=4, overlap=2, levels=2, cp1=4,
             cp2=4, cp3=2, nsteps=2, rtol=1e-11),
        # benchmark P8's grid G48 (6 x 48^2 x 72) in FP64 throughout: the reference arm of every accuracy claim
        dict(name='step_fp64_48x72', op='step', Ns=48, Nr=72, prec='fp64', p1=3, p2=3, p3=3, overlap=2, levels=2,
             nsteps=1, rtol=1e-8),
        # BF16 factors on a grid that no box edge divides evenly
        dict(name='step_bf16_50x46', op='step', Ns=50, Nr=46, prec='bf16', p1=2, p2=2, p3=3, overlap=2, levels=2,
             nsteps=2, rtol=1e-11),
        # the 9.4-million-cell shell: where memory traffic, not launches, sets the pace
        dict(name='step_fp32_128x96', op='step', Ns=128, Nr=96, prec='fp32', p1=4, p2=4, p3=6, overlap=2, levels=2,
             nsteps=1, rtol=1e-11),
        # one-level solve on an odd grid (no coarse mesh exists): the paper's one-level RAS rows
        dict(name='solve_ppbe_fp64_45x39', op='solve', kind='ppbe', Ns=45, Nr=39, prec='fp64', p1=2, p2=2, p3=3,
             overlap=1, levels=1, rtol=1e-8),
        # many right-hand sides on uneven boxes: how the learned correction's training targets are made
        dict(name='batch_ppbe_fp64_24', op='batch', kind='ppbe', Ns=24, Nr=24, prec='fp64', nrhs=8, overlap=1, rtol=1e-6),
        # operator applies alone: the outer solve's, the inner solves' at full size, a small ragged one
        dict(name='apply_vtbe_fp64_64', op='apply', kind='vtbe', Ns=64, Nr=64, prec='fp64', **_boxes(64, 64)),
        dict(name='apply_vtbe_fp32_128x96', op='apply', kind='vtbe', Ns=128, Nr=96, prec='fp32', **_boxes(128, 96)),
        dict(name='apply_ppbe_fp32_33x17', op='apply', kind='ppbe', Ns=33, Nr=17, prec='fp32', **_boxes(33, 17)),
        # the learned correction: inference once per coarse solve, and one training batch's gradient
        dict(name='net_forward_32', op='net', Ns=32, Nr=32, C=16, levels=3, nb=1, grad=False),
        dict(name='net_grad_32', op='net', Ns=32, Nr=32, C=16, levels=3, nb=8, grad=True),
    ]


def draw(rng):
    def size(lo, hi, mult=1):
        return mult * round(math.exp(rng.uniform(math.log(lo / mult), math.log(hi / mult))))

    op = rng.choice(['step', 'step', 'apply', 'apply', 'solve', 'batch', 'net'])
    if op == 'step':
        prec = rng.choice(['fp64', 'fp32', 'fp32', 'bf16'])
        Ns, Nr = size(12, 64 if prec == 'fp64' else 100, 2), size(12, 64 if prec == 'fp64' else 96, 2)
        levels = 1 if Ns < 16 or Nr < 16 else 2
        return dict(op=op, Ns=Ns, Nr=Nr, prec=prec, overlap=rng.choice([1, 2]), levels=levels, nsteps=rng.choice([1, 2]),
                    rtol=1e-8 if prec == 'fp64' else 1e-11, **_boxes(Ns, Nr))
    if op == 'apply':
        Ns, Nr = size(8, 128), size(6, 128)
        return dict(op=op, kind=rng.choice(['vtbe', 'ppbe']), Ns=Ns, Nr=Nr, prec=rng.choice(['fp64', 'fp32']),
                    **_boxes(Ns, Nr))
    if op == 'solve':
        Ns, Nr, levels = size(10, 56), size(8, 56), rng.choice([1, 1, 2])
        if levels == 2:
            Ns, Nr = Ns // 2 * 2, Nr // 2 * 2
        return dict(op=op, kind=rng.choice(['vtbe', 'ppbe']), Ns=Ns, Nr=Nr, prec='fp64', overlap=rng.choice([1, 2]),
                    levels=levels, rtol=1e-8, **_boxes(Ns, Nr))
    if op == 'batch':
        return dict(op=op, kind=rng.choice(['vtbe', 'ppbe']), Ns=size(12, 36, 4), Nr=size(12, 36, 4), prec='fp64',
                    nrhs=rng.choice([1, 3, 4, 8, 13]), overlap=rng.choice([1, 2]), rtol=1e-6)
    levels = rng.choice([1, 2, 3])
    return dict(op=op, Ns=size(8, 40, 1 << levels), Nr=size(8, 40, 1 << levels), C=rng.choice([16, 32]), levels=levels,
                nb=rng.choice([1, 2, 4]), grad=rng.random() < 0.5)


# ---------------------------------------------------------------- handles a program keeps
_plans = weakref.WeakValueDictionary()


def _dt(case):
    """The steps bench.py's shells take at their CFL limit, scaled to this grid."""
    return min(1e-4, 3.6e-3 / max(case['Ns'], case['Nr']))


class Plan:
    """Grid, systems, time-stepping state or network of one case; every prepared input of the case uses it."""

    def __init__(self, case):
        self.owned = []
        Ns, Nr, op = case['Ns'], case['Nr'], case['op']
        if op == 'net':
            self.net = self._own(fv.fv_net_create(case['C'], Ns, Nr, levels=case['levels'], max_batch=case['nb']),
                                 fv.fv_net_free)
            return
        self.grid = self._own(fv.fv_build_grid(Ns, Nr), fv.fv_free_grid)
        ph = dict(PHYS, dt=_dt(case))
        prec = PREC[case['prec']]
        mixed = {} if prec == fv.FV_PREC_FP64 else dict(precision=prec, inner_gs_passes=1)
        box = dict(p=(case.get('p1', 1), case.get('p2', 1), case.get('p3', 1)), overlap=case.get('overlap', 1))
        if op == 'step':
            inner = (dict(mixed, inner_maxit=4), dict(mixed, inner_maxit=8, coarse_maxit=10)) if mixed else ({}, {})
            coarse = dict(levels=case['levels'], coarse_p=(case.get('cp1', 0), case.get('cp2', 0), case.get('cp3', 0)))
            self.V = self._own(fv.fv_assemble_system(self.grid, fv.FV_VTBE, **ph, **box, **inner[0]), fv.fv_free_system)
            self.P = self._own(fv.fv_assemble_system(self.grid, fv.FV_PPBE, **ph, **box, **coarse, **inner[1]),
                               fv.fv_free_system)
            zero = torch.zeros(9 * 6 * Ns * Ns * Nr, dtype=torch.float64, device='cuda')
            self.state = self._own(fv.fv_state_create(self.grid, zero, **ph), fv.fv_free_state)
            return
        if op == 'batch':
            box = dict(overlap=case['overlap'], boxes=uneven_boxes(Ns, Nr, sizes=(4, 8, 12), seed=1))
        self.system = self._own(fv.fv_assemble_system(self.grid, KIND[case['kind']], **ph, **box, **mixed,
                                                      levels=case.get('levels', 1)), fv.fv_free_system)

    def _own(self, handle, free):
        self.owned.append((handle, free))
        return handle

    def __del__(self):
        for handle, free in reversed(self.owned):
            free(handle)


def _plan(case):
    key = repr(sorted((k, v) for k, v in case.items() if k != 'name'))
    plan = _plans.get(key)
    if plan is None:
        plan = _plans[key] = Plan(case)
    return plan


# ---------------------------------------------------------------- inputs
def _rand(shape, seed):
    return torch.randn(shape, dtype=torch.float64, generator=torch.Generator().manual_seed(seed)).cuda()


def _noise(shape, seed):
    return torch.randn(shape, dtype=torch.float64, device='cuda', generator=torch.Generator('cuda').manual_seed(seed))


def _smooth(shell, d, seed):
    """d random quadratic polynomials of the position on the shell's cells, (d, 6, Nr, Ns, Ns)."""
    c = _rand((d, 10), seed)
    x, y, z = shell.x
    mono = (torch.ones_like(x), x, y, z, x * x, y * y, z * z, x * y, y * z, z * x)
    return torch.stack([sum(c[a, m] * mono[m] for m in range(10)) for a in range(d)])


def _fields(case, seed):
    """Seeded initial fields of the shells (9N values): Theta and u of size 1e-2 that vanish at the walls, u and the
    perturbation of B curls (divergence free), B the paper's benchmark field plus that perturbation; P = P_b = 0."""
    s = Shell(case['Ns'], case['Nr'])
    x = s.x
    r = s.r.view(1, -1, 1, 1).expand(6, -1, s.Ns, s.Ns)
    b, db = (r - RI) * (RO - r), RI + RO - 2 * r
    A = _rand((2, 3, 4), seed)

    def curl(m):  # curl(b^2 a) for a(x) = M x + c: grad(b^2) x a + b^2 curl a
        a = [m[i, 0] * x[0] + m[i, 1] * x[1] + m[i, 2] * x[2] + m[i, 3] for i in range(3)]
        g = [2 * b * db * x[i] / r for i in range(3)]
        w = (m[2, 1] - m[1, 2], m[0, 2] - m[2, 0], m[1, 0] - m[0, 1])
        v = torch.stack([g[(i + 1) % 3] * a[(i + 2) % 3] - g[(i + 2) % 3] * a[(i + 1) % 3] + b * b * w[i] for i in range(3)])
        return 1e-2 * v / v.abs().max()

    th, ph = torch.arccos((x[2] / r).clamp(-1, 1)), torch.atan2(x[1], x[0])
    Br = 5 / 8 * (9 * r ** 3 - 4 * (4 + 3 * (RI + RO)) * r ** 2 + (4 * RO + RI * (4 + 3 * RO)) * 6 * r - 48 * RI * RO) / r
    Br, Bt = Br * th.cos(), -15 / 4 * (r - RI) * (r - RO) * (3 * r - 4) / r * th.sin()
    Bp = 15 / 8 * torch.sin(math.pi * (r - RI)) * torch.sin(2 * th)
    B0 = torch.stack([Br * th.sin() * ph.cos() + Bt * th.cos() * ph.cos() - Bp * ph.sin(),
                      Br * th.sin() * ph.sin() + Bt * th.cos() * ph.sin() + Bp * ph.cos(), Br * th.cos() - Bt * th.sin()])
    T = b * _smooth(s, 1, seed + 1)[0]
    out = torch.zeros(9, 6, s.Nr, s.Ns, s.Ns, dtype=torch.float64, device='cuda')
    out[0:3], out[3], out[4:7] = curl(A[0]), 1e-2 * T / T.abs().max(), B0 + curl(A[1])
    return out.reshape(-1)


def _net_params(case, seed):
    """He-initialised weights, layer by layer as include/fv_net.h lays them out."""
    rng = np.random.default_rng(seed)
    return np.concatenate([np.concatenate([rng.standard_normal(27 * ci * co) * math.sqrt(2 / (27 * ci)),
                                           0.05 * rng.standard_normal(co)]) for ci, co in _layers(case)]).astype(np.float32)


def _layers(case):
    C, L = case['C'], case['levels']
    return [(2 if m == 0 else C, C) for m in range(2 * (L + 1))] + [(2 * C, C)] * L + [(C, 2)]


def _net_vectors(case, seed):
    """Coarse right-hand sides and corrections: noise smoothed over a few cells, one row a sample."""
    n, nb = (2, 6, case['Nr'], case['Ns'], case['Ns']), case['nb']

    def field(sd):
        f = _noise((nb,) + n, sd)
        for ax in (3, 4, 5):
            f = 0.5 * f + 0.25 * (f.roll(1, ax) + f.roll(-1, ax))
        return f.reshape(nb, -1).contiguous()
    return field(seed), 0.3 * field(seed + 1)


def _solution(case, seed, d):
    """A solution (smooth, with a little noise) for manufactured right-hand sides, and the operator's shell."""
    s = Shell(case['Ns'], case['Nr'])
    x = _smooth(s, d, seed)
    return s, x + 1e-3 * _noise(x.shape, seed + 7)


class State:
    pass


def prepare(case, seed):
    st = State()
    st.case, st.plan = case, _plan(case)
    op = case['op']
    if op == 'step':
        st.init = _fields(case, seed)
        st.out = torch.empty_like(st.init)
    elif op == 'net':
        fv.fv_net_set_params(st.plan.net, _net_params(case, 11))
        st.r, st.e = _net_vectors(case, seed)
        st.out = torch.empty_like(st.r)
    else:
        d = 7 if case['kind'] == 'vtbe' else 2
        n = d * 6 * case['Ns'] ** 2 * case['Nr']
        if op == 'apply':
            st.x = _noise((n,), seed)
            if case['prec'] == 'fp32':
                st.x = st.x.float()
            st.out = torch.empty_like(st.x)
        else:
            rows = []
            for q in range(case.get('nrhs', 1)):
                s, x = _solution(case, seed + 100 * q, d)
                rows.append(s.apply(case['kind'], x, _dt(case)).reshape(-1))
            st.b = torch.stack(rows) if op == 'batch' else rows[0]
            st.out = torch.empty_like(st.b)
    return st


def run(st):
    c, p, op = st.case, st.plan, st.case['op']
    if op == 'step':
        fv.fv_state_reset(p.state, st.init)
        fv.fv_time_step(p.state, p.V, p.P, nsteps=c['nsteps'], rtol=c['rtol'])
        return fv.fv_state_get(p.state, st.out)  # u, Theta, B, P, P_b
    if op == 'net':
        if c['grad']:
            loss, g = fv.fv_net_loss_grad(p.net, c['nb'], st.r, st.e)
            return {'loss': loss, 'grad': g}
        return fv.fv_net_forward(p.net, c['nb'], st.r, st.out)
    if op == 'apply':
        return (fv.fv_apply_op if c['prec'] == 'fp64' else fv.fv_apply_op_fp32)(p.system, st.x, st.out)
    st.out.zero_()  # x0 = 0
    (fv.fv_gmres_solve_batch if op == 'batch' else fv.fv_gmres_solve)(p.system, st.b, st.out, rtol=c['rtol'])
    d, rows = 7 if c['kind'] == 'vtbe' else 2, st.out.view(c.get('nrhs', 1), -1)
    N = rows.shape[1] // d
    return [rows[:, :N], rows[:, N:]]


def work(case):
    N = 6 * case['Ns'] ** 2 * case['Nr']
    op = case['op']
    if op == 'step':  # the fields in and out
        return dict(bytes=2 * 9 * 8 * N * case['nsteps'], flops=0)
    if op == 'net':
        flops = sum(2 * 27 * ci * co * (N >> 3 * l) for (ci, co), l in zip(_layers(case), _layer_levels(case)))
        return dict(bytes=(2 if not case['grad'] else 4) * 2 * 8 * N * case['nb'],
                    flops=case['nb'] * flops * (3 if case['grad'] else 1))
    d = 7 if case['kind'] == 'vtbe' else 2
    if op == 'apply':  # x in, y out; 9 horizontal and 3 radial terms a row
        return dict(bytes=2 * d * N * (8 if case['prec'] == 'fp64' else 4), flops=2 * 12 * d * N)
    return dict(bytes=2 * d * 8 * N * case.get('nrhs', 1), flops=0)


def _layer_levels(case):
    L = case['levels']
    return [m // 2 for m in range(2 * (L + 1))] + list(range(L - 1, -1, -1)) + [0]


# ---------------------------------------------------------------- what the calls should return
def exact(case, seed):
    op = case['op']
    if op == 'step':  # both linear systems would have to be solved to round-off without a preconditioner: minutes
        return None
    if op == 'net':
        return _net_exact(case, seed)
    d = 7 if case['kind'] == 'vtbe' else 2
    if op == 'apply':
        x = _noise((d * 6 * case['Ns'] ** 2 * case['Nr'],), seed)
        x = x.float().double() if case['prec'] == 'fp32' else x
        s = Shell(case['Ns'], case['Nr'])
        return s.apply(case['kind'], x.view(d, 6, s.Nr, s.Ns, s.Ns), _dt(case)).reshape(-1)
    rows = torch.stack([_solution(case, seed + 100 * q, d)[1].reshape(-1) for q in range(case.get('nrhs', 1))])
    N = rows.shape[1] // d
    return [rows[:, :N] if case['kind'] == 'vtbe' else None, rows[:, N:]]  # P is determined up to a constant


_M = np.array([[[1, 0, 0], [0, 1, 0], [0, 0, 1]], [[0, -1, 0], [1, 0, 0], [0, 0, 1]], [[-1, 0, 0], [0, -1, 0], [0, 0, 1]],
               [[0, 1, 0], [-1, 0, 0], [0, 0, 1]], [[0, 0, -1], [0, 1, 0], [1, 0, 0]], [[0, 0, 1], [0, 1, 0], [-1, 0, 0]]],
              dtype=np.float64)


def _side_points(side, t, edge):
    return {0: (np.full_like(t, -edge), t), 1: (np.full_like(t, edge), t), 2: (t, np.full_like(t, -edge)),
            3: (t, np.full_like(t, edge))}[side]


def _dirs(p, xi, eta):
    v = np.stack([np.ones_like(xi), np.tan(xi), np.tan(eta)], -1)
    return (v / np.linalg.norm(v, axis=-1, keepdims=True)) @ _M[p].T


class Shell:
    """The cubed-sphere shell's operators in plain torch (FP64): six panels padded by one ghost layer (quadratic
    interpolation along the neighbour's first grid line, panel-edge faces the mean of the two panels' fluxes)."""

    def __init__(self, Ns, Nr):
        cu = lambda a: torch.tensor(a, dtype=torch.float64, device='cuda')  # noqa: E731
        self.Ns, self.Nr, self.hs, self.hr = Ns, Nr, math.pi / (2 * Ns), (RO - RI) / Nr
        hs, hr = self.hs, self.hr
        c, f = -math.pi / 4 + (np.arange(Ns) + 0.5) * hs, -math.pi / 4 + np.arange(Ns + 1) * hs
        self.r = cu(RI + (np.arange(Nr) + 0.5) * hr)
        self.rf = cu(RI + np.arange(Nr + 1) * hr)

        def metric(xi, eta):  # [eta][xi]: sigma, sqrt(g) g^11, g^22, g^12 over r^2, 1, 1, 1
            X, Y = np.tan(xi)[None, :], np.tan(eta)[:, None]
            s = np.sqrt(1 + X * X + Y * Y)
            return [cu(a + 0 * (X + Y)) for a in ((1 + X * X) * (1 + Y * Y) / s ** 3, (1 + Y * Y) / s, (1 + X * X) / s,
                                                  X * Y / s)]
        self.sigma = metric(c, c)[0]
        _, self.fx, _, self.fxc = metric(f, c)
        _, _, self.fy, self.fyc = metric(c, f)
        xi, eta = np.meshgrid(c, c, indexing='xy')
        self.rhat = cu(np.stack([_dirs(p, xi, eta) for p in range(6)])).permute(3, 0, 1, 2)  # [3][p][j][i]
        self.x = self.rhat[:, :, None] * self.r.view(1, 1, -1, 1, 1)
        self.edges = {}
        for p in range(6):
            for side in range(4):
                g, e = _dirs(p, *_side_points(side, c, math.pi / 4 + hs / 2)), _dirs(p, *_side_points(side, c, math.pi / 4))
                q = max(range(6), key=lambda k: float((g @ _M[k])[0, 0]))
                loc, le = g @ _M[q], e @ _M[q]
                a, b = np.arctan(loc[:, 1] / loc[:, 0]), np.arctan(loc[:, 2] / loc[:, 0])
                lim = math.pi / 4 - hs / 2
                sq = int(np.argmin([np.abs(a + lim).max(), np.abs(a - lim).max(), np.abs(b + lim).max(), np.abs(b - lim).max()]))
                tau, te = (b, np.arctan(le[:, 2] / le[:, 0])) if sq < 2 else (a, np.arctan(le[:, 1] / le[:, 0]))
                frac = (tau + math.pi / 4) / hs - 0.5
                m = np.clip(np.floor(frac + 0.5).astype(int), 1, Ns - 2)
                s = frac - m
                w = np.stack([0.5 * s * (s - 1), 1 - s * s, 0.5 * s * (s + 1)])
                tm = np.rint((te + math.pi / 4) / hs - 0.5).astype(int)
                self.edges[p, side] = (q, sq, torch.tensor(np.stack([m - 1, m, m + 1]), device='cuda'), cu(w),
                                       torch.tensor(tm, device='cuda'), 1.0 if (side % 2) != (sq % 2) else -1.0)

    @staticmethod
    def line(a, side, ring=0):
        """The row or column of [..., j, i] next to `side` (ring = 1: of a padded array, the ghosts)."""
        lo, hi, inner = (0, -1, slice(1, -1)) if ring else (0, -1, slice(None))
        return {0: a[..., inner, lo], 1: a[..., inner, hi], 2: a[..., lo, inner], 3: a[..., hi, inner]}[side]

    def pad(self, x, walls):
        """[c][p][k][j][i] -> one ghost layer on every side; walls: a rule per component ('odd', 'even', or 'B')."""
        out = torch.zeros(x.shape[0], 6, self.Nr + 2, self.Ns + 2, self.Ns + 2, dtype=torch.float64, device='cuda')
        out[:, :, 1:-1, 1:-1, 1:-1] = x
        for (p, side), (q, sq, m, w, _, _) in self.edges.items():
            ln = self.line(x[:, q], sq)
            self.line(out[:, p, 1:-1], side, 1).copy_(sum(w[a] * ln[..., m[a]] for a in range(3)))
        for j, jn in ((0, 1), (-1, -2)):
            for i, im in ((0, 1), (-1, -2)):
                out[..., j, i] = out[..., jn, i] + out[..., j, im] - out[..., jn, im]
        inner = (slice(1, -1), slice(1, -1))
        for kk, kc, rw in ((0, 0, RI), (-1, -1, RO)):
            rc = float(self.r[kc])
            for c, rule in enumerate(walls):
                out[(c, slice(None), kk) + inner] = (1 if rule == 'even' else -1) * x[c, :, kc]
            if 'B' in walls:
                b = walls.index('B')
                dot = (x[b:b + 3, :, kc] * self.rhat).sum(0)
                out[(slice(b, b + 3), slice(None), kk) + inner] += (1 + (rc / (2 * rw - rc)) ** 2) * dot * self.rhat
        return out

    def laplacian(self, x, walls):
        hs, hr = self.hs, self.hr
        P = self.pad(x, walls)
        h = P[:, :, 1:-1]
        dy, dx = h[..., 2:, :] - h[..., :-2, :], h[..., 2:] - h[..., :-2]
        fx = self.fx * hr * (h[..., 1:-1, 1:] - h[..., 1:-1, :-1]) + self.fxc * hr / 4 * (dy[..., 1:] + dy[..., :-1])
        fy = self.fy * hr * (h[..., 1:, 1:-1] - h[..., :-1, 1:-1]) + self.fyc * hr / 4 * (dx[..., 1:, :] + dx[..., :-1, :])
        ends = {k: self.line(fx if k[1] < 2 else fy, k[1])[:, k[0]].clone() for k in self.edges}
        for (p, side), (q, sq, _, _, tm, sg) in self.edges.items():
            self.line(fx if side < 2 else fy, side)[:, p] = 0.5 * (ends[p, side] + sg * ends[q, sq][..., tm])
        v = P[:, :, :, 1:-1, 1:-1]
        fr = self.sigma * hs * hs * (self.rf ** 2).view(-1, 1, 1) * (v[:, :, 1:] - v[:, :, :-1]) / hr
        div = fx[..., 1:] - fx[..., :-1] + fy[..., 1:, :] - fy[..., :-1, :] + fr[:, :, 1:] - fr[:, :, :-1]
        return div / (self.sigma * (self.r ** 2).view(-1, 1, 1) * hs * hs * hr)

    def apply(self, kind, x, dt):
        E, Ra, Pr, Pm = (PHYS[k] for k in ('E', 'Ra', 'Pr', 'Pm'))
        if kind == 'ppbe':
            return dt / (2 * E) * self.laplacian(x, ['even', 'odd'])
        L = self.laplacian(x, ['odd'] * 4 + ['B'] * 3)
        L[3] /= Pr
        L[4:] /= Pm
        L[0] += 2 / E * x[1]
        L[1] -= 2 / E * x[0]
        L[:3] += Ra / (E * RO) * x[3] * self.x
        L[3] += RI * RO / (self.r ** 3).view(-1, 1, 1) * (x[:3] * self.x).sum(0)
        return x - dt / 2 * L


def _net_exact(case, seed):
    """The U-Net of include/fv_net.h and its loss in FP64 (27 shifted products a convolution)."""
    par = torch.tensor(_net_params(case, 11).astype(np.float64), device='cuda', requires_grad=bool(case['grad']))
    W, off = [], 0
    for ci, co in _layers(case):
        w = par[off:off + 27 * ci * co].view(co, ci, 27)
        W.append((w, par[off + 27 * ci * co:off + 27 * ci * co + co]))
        off += 27 * ci * co + co
    edges = {}

    def conv(a, m):  # a: [b][c][p][z][y][x]
        n, Z = a.shape[-1], a.shape[3]
        if n not in edges:  # the pairing of a finer grid's edge faces, four to one
            edges[n] = {k: (e[0], e[1], (e[4][::4] // 4)) for k, e in Shell(4 * n, 2).edges.items()}
        z = torch.zeros(a.shape[:3] + (Z + 2, n + 2, n + 2), dtype=torch.float64, device='cuda')
        z[:, :, :, 1:-1, 1:-1, 1:-1] = a
        for (p, side), (q, sq, tm) in edges[n].items():
            Shell.line(z[:, :, p, 1:-1], side, 1).copy_(Shell.line(a[:, :, q], sq)[..., tm])
        w, b = W[m]
        y = sum(torch.einsum('oc,bcpzyx->bopzyx', w[:, :, 9 * dz + 3 * dy + dx],
                             z[:, :, :, dz:dz + Z, dy:dy + n, dx:dx + n])
                for dz in range(3) for dy in range(3) for dx in range(3))
        return y + b.view(1, -1, 1, 1, 1, 1)

    def pool(a):
        return a.unflatten(5, (-1, 2)).mean(6).unflatten(4, (-1, 2)).mean(5).unflatten(3, (-1, 2)).mean(4)

    def up(a):
        return a.repeat_interleave(2, 3).repeat_interleave(2, 4).repeat_interleave(2, 5)

    with torch.set_grad_enabled(bool(case['grad'])):
        shape = (case['nb'], 2, 6, case['Nr'], case['Ns'], case['Ns'])
        r, e = (v.view(shape) for v in _net_vectors(case, seed))
        s = r.square().mean((1, 2, 3, 4, 5), keepdim=True).sqrt()
        L, a, E = case['levels'], r / s, []
        for l in range(L + 1):
            a = pool(a) if l else a
            a = torch.relu(conv(torch.relu(conv(a, 2 * l)), 2 * l + 1))
            E.append(a)
        for l in range(L - 1, -1, -1):
            a = torch.relu(conv(torch.cat([E[l], up(a)], 1), 2 * (L + 1) + L - 1 - l))
        y = conv(a, 3 * L + 2)
        if not case['grad']:
            return (s * y).reshape(case['nb'], -1)
        loss = (y - e / s).square().mean()
        loss.backward()
    return {'loss': float(loss.detach()), 'grad': par.grad}
