"""The work that a user of this library has it do, as measurable cases.

Boxes, populations and temperatures are those of the workloads in
``paper_2403_09158_gb300.workload`` and of the tests; every pass goes through the
ctypes binding, as a program that drives the library does.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2403_09158_gb300 import okmc as ok
from paper_2403_09158_gb300 import workload as wl

H = wl.VOXEL_NM
FE = (243.0, 145.0, 116.0)              # synthetic Fe constants of the mixed populations, GPa
FE_PAPER = (289.34, 152.34, 107.43)     # the paper's Table 1, used by the two-loop settings
KAPPA = 6.241509074                     # eV per GPa nm^3
KB = 8.617333262e-5                     # eV/K


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest replicas, in the accurate mode: short steps, bound by latency
        {'name': 'step_small_fp64', 'do': 'step', 'nx': 32, 'ny': 32, 'nz': 32, 'nd': 10, 'fp64': True, 'rmax': 1.0,
         'T': 300.0, 'steps': 10, 'fixed': False},
        # one solve for a caller that may not allocate device memory, at the largest box it takes
        {'name': 'static_solve_64', 'do': 'static', 'nx': 64, 'ny': 64, 'nz': 64, 'nd': 12},
        # a point of the loop-loop energy profile: move a loop, exact and dipole energies
        {'name': 'profile_128', 'do': 'profile', 'n': 128, 'radius': 3.3},
        # kinetics at the medium size: events one by one
        {'name': 'step_medium', 'do': 'step', 'nx': 128, 'ny': 128, 'nz': 128, 'nd': 200, 'fp64': False, 'rmax': 2.5,
         'T': 400.0, 'steps': 10, 'fixed': False},
        # the same box in the accurate mode: one defect moved, all site and candidate energies
        {'name': 'energies_medium_fp64', 'do': 'energies', 'nx': 128, 'ny': 128, 'nz': 128, 'nd': 200, 'fp64': True,
         'rmax': 2.5, 'moved': 1},
        # the headline workload: residence-time events in the dense 256^3 box
        {'name': 'step_large', 'do': 'step', 'nx': 256, 'ny': 256, 'nz': 256, 'nd': 2000, 'fp64': False, 'rmax': 4.0,
         'T': 500.0, 'steps': 5, 'fixed': False},
        # the stress field itself after every defect has moved (a full solve)
        {'name': 'solve_large', 'do': 'solve', 'nx': 256, 'ny': 256, 'nz': 256, 'nd': 2000, 'fp64': False, 'rmax': 4.0},
        # boxes with unequal edges
        {'name': 'solve_ragged', 'do': 'solve', 'nx': 96, 'ny': 64, 'nz': 160, 'nd': 30, 'fp64': False, 'rmax': 1.0},
        # the paper's two-loop kinetics in a box near its 500 a0
        {'name': 'kinetics_512', 'do': 'kinetics', 'n': 512, 'x_rel': 10.0, 'steps': 2},
        # a replica becoming resident: stencils, energy lists, self terms
        {'name': 'setup_large', 'do': 'setup', 'n': 256, 'nd': 2000, 'rmax': 4.0},
        # an ensemble of replicas of uneven edges advanced together
        {'name': 'ensemble_8', 'do': 'batch', 'edges': '64,96,128,160,192,128,96,64', 'steps': 3},
        # a loop's energy at continuous positions along its glide axis
        {'name': 'shift_128', 'do': 'shift', 'n': 128, 'm': 121, 'radius': 3.3, 'fp64': False},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _box(rng, edges, voxels):
    while True:
        n = [rng.choice(edges) for _ in range(3)]
        if n[0] * n[1] * n[2] <= voxels:
            return n


def draw(rng):
    do = rng.choice(['step', 'step', 'step64', 'static', 'profile', 'energies', 'solve', 'solve', 'kinetics', 'setup',
                     'batch', 'shift'])
    edges = [16, 32, 48, 64, 80, 96, 128, 144, 160, 192, 240, 256, 288, 320, 384, 400, 480, 512]
    if do == 'step':
        n = rng.choice([48, 64, 96, 128, 160, 192, 256])
        return {'do': 'step', 'nx': n, 'ny': n, 'nz': n, 'nd': max(2, int(_log_uniform(rng, 0.1, 1.0) * 2000 * (n / 256) ** 3)),
                'fp64': False, 'rmax': min(4.0, 0.07 * n), 'T': round(rng.uniform(300, 600), 2), 'steps': rng.randint(1, 5),
                'fixed': rng.random() < 0.3}
    if do == 'step64':
        n = rng.choice([32, 48, 64, 80, 96])
        return {'do': 'step', 'nx': n, 'ny': n, 'nz': n, 'nd': rng.randint(2, 10 + n // 4), 'fp64': True, 'rmax': 1.0,
                'T': round(rng.uniform(300, 600), 2), 'steps': rng.randint(1, 10), 'fixed': False}
    if do == 'static':
        while True:
            n = _box(rng, [16, 32, 48, 64, 80, 96, 128], 64 ** 3)
            if 6 * (n[0] // 2 + 1) * n[1] * n[2] <= 6 * 33 * 64 * 64:
                return {'do': 'static', 'nx': n[0], 'ny': n[1], 'nz': n[2], 'nd': rng.randint(1, 4)}
    if do == 'profile':
        return {'do': 'profile', 'n': rng.choice([96, 128, 160, 192, 256]), 'radius': round(rng.uniform(1.0, 4.0), 3)}
    if do == 'energies':
        n = _box(rng, [48, 64, 80, 96, 128, 144, 160], 128 ** 3)
        return {'do': 'energies', 'nx': n[0], 'ny': n[1], 'nz': n[2], 'nd': rng.randint(2, 40), 'fp64': True, 'rmax': 1.5,
                'moved': rng.randint(1, 2)}
    if do == 'solve':
        fp64 = rng.random() < 0.25
        n = _box(rng, edges, int(_log_uniform(rng, 32 ** 3, 128 ** 3 if fp64 else 256 ** 3)))
        return {'do': 'solve', 'nx': n[0], 'ny': n[1], 'nz': n[2], 'nd': rng.randint(2, 8), 'fp64': fp64,
                'rmax': min(1.5, 0.07 * min(n))}
    if do == 'kinetics':
        return {'do': 'kinetics', 'n': rng.choice([192, 256, 320, 384, 400, 480]), 'x_rel': round(rng.uniform(8, 20), 2),
                'steps': rng.randint(1, 2)}
    if do == 'setup':
        n = rng.choice([48, 64, 96, 128, 160, 192])
        return {'do': 'setup', 'n': n, 'nd': max(2, int(_log_uniform(rng, 0.1, 1.0) * 2000 * (n / 256) ** 3)),
                'rmax': min(4.0, 0.07 * n)}
    if do == 'batch':
        return {'do': 'batch', 'edges': ','.join(str(rng.choice([64, 96, 128, 160, 192])) for _ in range(rng.randint(2, 8))),
                'steps': rng.randint(1, 4)}
    return {'do': 'shift', 'n': rng.choice([64, 80, 96, 128]), 'm': rng.randint(1, 121), 'radius': round(rng.uniform(1, 3.3), 3),
            'fp64': rng.random() < 0.3}


# ------------------------------------------------------------------ inputs
def _dims(case):
    return (case['n'],) * 3 if 'n' in case else (case['nx'], case['ny'], case['nz'])


def _population(n, nd, seed, rmax):
    """The workloads' defect mix; the count falls until the box holds it."""
    while True:
        try:
            return wl.mixed_population(n, nd, seed, r111=(0.4, rmax), r100=(0.4, rmax))
        except RuntimeError:
            nd = max(1, int(nd * 0.9))


def _two_loops(n, x_rel, radius, seed):
    """The paper's pair of 1/2[111] loops, 10 nm apart across their glide axis (a quarter of
    the box where that is less), anywhere in the box."""
    w = wl.config_kinetics(x_rel, n=n, R_nm=radius, z_rel_nm=min(10.0, 0.25 * n * H))
    d = w.defects.copy()
    d['pos'] = np.mod(d['pos'] + 2 * np.random.default_rng(seed).integers(0, n, 3), 2 * n)
    return d


def _defects(case, seed):
    if case['do'] in ('kinetics', 'profile', 'shift'):
        n = case['n']
        return _two_loops(n, min(case.get('x_rel', 5.0), 0.2 * n * H), case.get('radius', 3.3), seed)
    return _population(_dims(case), case['nd'], seed, case.get('rmax', 0.6))


def _moved(d, n, count, seed):
    """Positions after a jump of `count` defects along their axis (all of them: count = 0)."""
    rng = np.random.default_rng(seed + 1)
    p = d['pos'].astype(np.int32)
    who = np.arange(len(d)) if count == 0 else rng.choice(len(d), min(count, len(d)), replace=False)
    jump = 2 * rng.integers(0, 2, (len(who), 3), dtype=np.int32) - 1
    p[who] = np.mod(p[who] + jump, 2 * np.array(n, np.int32))
    return np.ascontiguousarray(p)


def _replicas(case, seed):
    out = []
    for k, e in enumerate(int(x) for x in case['edges'].split(',')):
        nd = min(400, wl.density_cap(e)) // 2
        out.append(((e,) * 3, _population((e,) * 3, nd, 1000 * seed + k, 2.5), 300.0 + 37.5 * k))
    return out


def _constants(case):
    return FE_PAPER if case['do'] in ('kinetics', 'profile') else FE


def _grid(case, d, seed):
    g = ok.Grid(_dims(case), H, *_constants(case), precision=ok.FP64_FIELDS if case.get('fp64') else ok.FP32_FIELDS, seed=seed)
    g.set_defects(d)
    return g


def _shift_points(case, seed):
    x = np.random.default_rng(seed + 2).uniform(-6.0, 6.0, case['m'])
    return x[:, None] * np.ones(3) / math.sqrt(3.0)


def prepare(case, seed):
    do, s = case['do'], {'case': case, 'seed': seed}
    if do == 'batch':
        s['grids'] = []
        s['T'] = []
        for n, d, T in _replicas(case, seed):
            g = ok.Grid(n, H, *FE, seed=seed)
            g.set_defects(d)
            s['grids'].append(g)
            s['T'].append(T)
        s['batch'] = ok.Batch(s['grids'])
        return s
    d, n = _defects(case, seed), _dims(case)
    if do == 'static':
        eps = _field(d, d['pos'], n).to(torch.float32)
        s.update(lib=ok.load(), eps=eps, sig=torch.empty_like(eps), n=(ctypes.c_int32 * 3)(*n))
        return s
    if do == 'setup':
        s['grid'] = ok.Grid(n, H, *FE, seed=seed)
        s['defects'] = d
        return s
    g = s['grid'] = _grid(case, d, seed)
    if do == 'solve':
        s['at'] = [_moved(d, n, 0, seed), np.ascontiguousarray(d['pos'].astype(np.int32))]
        s['out'] = torch.empty((6, n[2], n[1], n[0]), device='cuda', dtype=torch.float64 if case['fp64'] else torch.float32)
    elif do in ('energies', 'profile'):
        s['at'] = [_moved(d, n, case.get('moved', 1), seed), np.ascontiguousarray(d['pos'].astype(np.int32))]
        if do == 'profile':
            g.dipole_self_terms()
    elif do == 'shift':
        s['X'] = d['pos'][0] * (0.5 * H) + _shift_points(case, seed)
    return s


def _next(s):
    """The two configurations in turn, so that every pass brings positions that are new to the grid."""
    p = s['at'][0]
    s['at'].reverse()
    return p


def run(s):
    case, do, g = s['case'], s['case']['do'], s.get('grid')
    if do == 'step':
        st = g.step(case['T'], case['steps'], mode=ok.FIXED_DT if case['fixed'] else ok.RESIDENCE)
        return {'positions': g.get_positions(), 'stats': st}
    if do == 'kinetics':
        st = g.step(300.0, case['steps'], mode=ok.FIXED_DT)
        return {'positions': g.get_positions(), 'stats': st}
    if do == 'batch':
        st = s['batch'].step(s['T'], case['steps'])
        return {'positions': [x.get_positions() for x in s['grids']], 'stats': st}
    if do == 'static':
        rc = s['lib'].okmc_solve_stress_static(s['eps'].data_ptr(), s['sig'].data_ptr(), s['n'], *FE, ok.MEAN_STRESS_ZERO,
                                               torch.cuda.current_stream().cuda_stream)
        if rc != ok.OKMC_OK:
            raise RuntimeError('okmc_solve_stress_static: %d' % rc)
        return {'stress': s['sig']}
    if do == 'setup':
        g.set_defects(s['defects'])
        return {'self_terms': g.self_terms()}
    if do == 'shift':
        return {'energies': g.shift_energies(0, s['X'])}
    g.set_positions(_next(s))
    if do == 'solve':
        return {'stress': g.solve_stress(out=s['out'])}
    if do == 'profile':
        e, ec = g.dipole_energies()
        return {'site': g.interaction_energies(), 'dipole': e, 'dipole_jumps': ec}
    return {'site': g.interaction_energies(), 'jumps': g.candidate_energies()[0]}


def work(case):
    """One pass: the eigenstrain read and the stress written once per solve; the flops of the
    six forward and six inverse real transforms and of the Green operator.  A set-up reads
    a type table and writes the field once; a shift reads the eigenstrain."""
    if case['do'] == 'batch':
        boxes, w = [int(x) ** 3 for x in case['edges'].split(',')], 4
    else:
        n = _dims(case)
        boxes, w = [n[0] * n[1] * n[2]], 8 if case.get('fp64') else 4
    solves = case.get('steps', 1)
    N = sum(boxes)
    transform = sum(2.5 * b * math.log2(b) for b in boxes)
    if case['do'] == 'setup':
        return {'bytes': 6 * N * w, 'flops': 2 * transform}
    if case['do'] == 'shift':
        return {'bytes': 6 * N * w, 'flops': 8 * transform + 0.5 * N * (300 + 10 * case['m'])}
    return {'bytes': solves * 12 * N * w, 'flops': solves * (12 * transform + 0.5 * N * 200)}


# ------------------------------------------------------------------ the same results in 64 bits
# The paper's formulas (eigenstrains of Sec. 3.1 on the voxels of Sec. 3.4, the solve of
# Sec. 3.2 by complex transforms, the energies of Sec. 2) written out with torch.
def _geometry(d):
    """(e (6), alpha-free volume / h^3, inside test, scan half-width)."""
    if int(d['type']) == wl.SIA_CLUSTER:
        rho3 = max(1.0, 3.0 * int(d['size']) / (8.0 * math.pi))
        v = 4.0 * math.pi / 3.0 * rho3
        e = 0.75 * int(d['size']) / (3.0 * v)
        return np.array([e, e, e, 0, 0, 0.]), v, (lambda x, y, z: (x * x + y * y + z * z) ** 3 <= 262144.0 * (rho3 * rho3)), \
            math.ceil(rho3 ** (1 / 3)) + 1
    if int(d['type']) == wl.LOOP_111:
        a = [1, 1, 1]
        if int(d['axis']):
            a[int(d['axis']) - 1] = -1
        b = math.sqrt(3.0) / 2
    else:
        a = [int(k == int(d['axis'])) for k in range(3)]
        b = 1.0
    a2, r = sum(x * x for x in a), float(d['radius_nm']) / H

    def inside(x, y, z):
        s = a[0] * x + a[1] * y + a[2] * z
        return (s * s <= 16 * a2) & (a2 * (x * x + y * y + z * z) - s * s <= a2 * (8.0 * float(d['radius_nm']) / H) ** 2)
    e = np.array([a[0] * a[0], a[1] * a[1], a[2] * a[2], a[1] * a[2], a[0] * a[2], a[0] * a[1]]) * (b / a2)
    return e, math.pi * r * r, inside, math.ceil(r) + 1


_STENCILS = {}


def _stencil(d, c):
    """(offsets (k, 3) in x, y, z; weights (k); eigenstrain (6)) of a defect in site class c."""
    key = (int(d['type']), int(d['axis']), int(d['size']), float(d['radius_nm']), c)
    if key not in _STENCILS:
        e, vol, inside, E = _geometry(d)
        s = (8 * np.arange(-E, E + 1)[:, None] + 2 * np.arange(4) + 1 - 4 * c).ravel().astype(np.float64)
        x = torch.from_numpy(s).cuda()
        k = len(s) // 4
        cnt = inside(x[:, None, None], x[None, :, None], x[None, None, :]).view(k, 4, k, 4, k, 4).sum(dim=(1, 3, 5))
        off = torch.nonzero(cnt)
        w = cnt[off[:, 0], off[:, 1], off[:, 2]].double()
        _STENCILS[key] = (off - E, w * (vol / w.sum()), torch.from_numpy(e).cuda())
    return _STENCILS[key]


def _voxels(off, base, n):
    v = [torch.remainder(off[:, a] + int(base[a]), n[a]) for a in range(3)]
    return (v[2] * n[1] + v[1]) * n[0] + v[0]


def _field(d, pos, n):
    eps = torch.zeros((6, n[0] * n[1] * n[2]), dtype=torch.float64, device='cuda')
    for k in range(len(d)):
        off, w, e = _stencil(d[k], int(pos[k][0]) & 1)
        eps.index_add_(1, _voxels(off, np.asarray(pos[k]) // 2, n), e[:, None] * w[None, :])
    return eps.view(6, n[2], n[1], n[0])


def _green(e, n, z, C):
    """Stress of the transformed eigenstrain e (6 x one z-plane) at that plane's frequencies."""
    f = [torch.fft.fftfreq(k, dtype=torch.float64, device='cuda') for k in n]
    q = [f[0][None, :], f[1][:, None], f[2][z].view(1, 1)]
    q = [x.expand(n[1], n[0]) for x in q]
    C11, C12, C44 = C
    tr = C12 * (e[0] + e[1] + e[2])
    t = [tr + (C11 - C12) * e[a] for a in range(3)] + [2 * C44 * e[a] for a in (3, 4, 5)]
    v = [q[0] * t[0] + q[1] * t[5] + q[2] * t[4], q[0] * t[5] + q[1] * t[1] + q[2] * t[3], q[0] * t[4] + q[1] * t[3] + q[2] * t[2]]
    cq = C44 * (q[0] ** 2 + q[1] ** 2 + q[2] ** 2)
    k = [cq + (C11 - C44) * q[a] ** 2 for a in range(3)]
    k12, k02, k01 = [(C12 + C44) * q[a] * q[b] for a, b in ((1, 2), (0, 2), (0, 1))]
    i00, i11, i22 = k[1] * k[2] - k12 ** 2, k[0] * k[2] - k02 ** 2, k[0] * k[1] - k01 ** 2
    i01, i02, i12 = k02 * k12 - k01 * k[2], k01 * k12 - k02 * k[1], k01 * k02 - k[0] * k12
    det = k[0] * i00 + k01 * i01 + k02 * i02
    if z == 0:
        det[0, 0] = 1.0
    w = [(i00 * v[0] + i01 * v[1] + i02 * v[2]) / det, (i01 * v[0] + i11 * v[1] + i12 * v[2]) / det,
         (i02 * v[0] + i12 * v[1] + i22 * v[2]) / det]
    qw = C12 * (q[0] * w[0] + q[1] * w[1] + q[2] * w[2])
    out = [qw + (C11 - C12) * q[a] * w[a] - t[a] for a in range(3)]
    out += [C44 * (q[a] * w[b] + q[b] * w[a]) - t[c] for c, a, b in ((3, 1, 2), (4, 0, 2), (5, 0, 1))]
    if z == 0:
        for x in out:
            x[0, 0] = 0.0
    return out


def _solve(eps, n, C):
    s = torch.empty_like(eps, dtype=torch.complex128)
    for a in range(6):
        s[a] = torch.fft.fftn(eps[a])
    for z in range(n[2]):
        for a, x in enumerate(_green([s[a, z].clone() for a in range(6)], n, z, C)):
            s[a, z] = x
    return torch.stack([torch.fft.ifftn(s[a]).real for a in range(6)])


_JUMPS = np.array([[1 if j & 4 else -1, 1 if j & 2 else -1, 1 if j & 1 else -1] for j in range(8)])
_DOUBLE = torch.tensor([1., 1, 1, 2, 2, 2], dtype=torch.float64)


def _sum_at(d, Y, sig, n):
    """-kappa h^3 times the sum of the defect's eigenstrain at Y against the stress."""
    off, w, e = _stencil(d, int(Y[0]) & 1)
    return -KAPPA * H ** 3 * ((e * _DOUBLE.cuda()) @ sig.view(6, -1)[:, _voxels(off, np.asarray(Y) // 2, n)]) @ w


class _SelfTerms:
    """W(c, k) of a defect against its own field, by the real-space kernel of its tensor."""

    def __init__(self, n, C):
        self.n, self.C, self.kernels, self.tables = n, C, {}, {}

    def kernel(self, e):
        unit = tuple(np.round((e / e.abs().max()).cpu().numpy(), 9))
        if unit not in self.kernels:
            n, E = self.n, e / e.abs().max()
            Q = torch.empty((n[2], n[1], n[0]), dtype=torch.float64, device='cuda')
            for z in range(n[2]):
                s = _green([E[a].expand(n[1], n[0]) for a in range(6)], n, z, self.C)
                Q[z] = sum(float(_DOUBLE[a]) * E[a] * s[a] for a in range(6))
            self.kernels[unit] = torch.fft.ifftn(Q).real.reshape(-1)
        return self.kernels[unit]

    def table(self, d):
        key = (int(d['type']), int(d['axis']), int(d['size']), float(d['radius_nm']))
        if key not in self.tables:
            n, st = self.n, [_stencil(d, c) for c in (0, 1)]
            K, s2 = self.kernel(st[0][2]), float(st[0][2].abs().max()) ** 2
            W = torch.empty((2, 9), dtype=torch.float64, device='cuda')
            for c in (0, 1):
                for k in range(9):
                    cp = c if k == 0 else 1 - c
                    shift = np.zeros(3, int) if k == 0 else (c + _JUMPS[k - 1]) // 2
                    (oa, wa, _), (ob, wb, _) = st[c], st[cp]
                    v = [torch.remainder(ob[None, :, a] + int(shift[a]) - oa[:, None, a], n[a]) for a in range(3)]
                    W[c, k] = -KAPPA * H ** 3 * s2 * (wa @ K[(v[2] * n[1] + v[1]) * n[0] + v[0]] @ wb)
            self.tables[key] = W
        return self.tables[key]


def _energies(d, pos, n, C, self_terms, jumps=True, sig=None):
    sig = _solve(_field(d, pos, n), n, C) if sig is None else sig
    E = []
    for k in range(len(d)):
        c, W = int(pos[k][0]) & 1, self_terms.table(d[k])
        at = [pos[k]] + ([pos[k] + j for j in _JUMPS] if jumps else [])
        E.append(torch.stack([_sum_at(d[k], Y, sig, n) - W[c, i] for i, Y in enumerate(at)]))
    E = torch.stack(E).cpu().numpy()
    return E[:, 0], E[:, 1:]


def _philox(step, who, tag, seed):
    x, k = [step & 0xFFFFFFFF, step >> 32, who, tag], [seed & 0xFFFFFFFF, seed >> 32]
    for r in range(10):
        if r:
            k = [(k[0] + 0x9E3779B9) & 0xFFFFFFFF, (k[1] + 0xBB67AE85) & 0xFFFFFFFF]
        p, q = 0xD2511F53 * x[0], 0xCD9E8D57 * x[2]
        x = [(q >> 32) ^ x[1] ^ k[0], q & 0xFFFFFFFF, (p >> 32) ^ x[3] ^ k[1], p & 0xFFFFFFFF]
    return [(((x[i + 1] << 21) | (x[i] >> 11)) + 1) * 2.0 ** -53 for i in (0, 2)]


def _allowed(d):
    if int(d['mobility']) == wl.THREE_D:
        return list(range(8))
    if int(d['mobility']) != wl.ONE_D:
        return []
    a = int(d['axis'])
    j = 4 * (a != 1) + 2 * (a != 2) + (a != 3)
    return [j, 7 - j]


def _residence(d, n, T, steps, seed, C):
    """The kinetic clock and last time step after residence-time events."""
    W, pos, clock, dt = _SelfTerms(n, C), d['pos'].astype(np.int64), 0.0, 0.0
    for step in range(steps):
        E, Ec = _energies(d, pos, n, C, W)
        line, total = [], 0.0
        for i in range(len(d)):
            al = _allowed(d[i])
            for j in sorted(al):
                r = 1e13 / len(al) * math.exp(-(float(d[i]['Em_eV']) + 0.5 * (Ec[i, j] - E[i])) / (KB * T))
                total += r
                line.append((total, i, j))
        u1, u2 = _philox(step, 0xFFFFFFFF, 0, seed)
        _, i, j = next((x for x in line if x[0] >= u1 * total), line[-1])
        pos[i] = np.mod(pos[i] + _JUMPS[j], 2 * np.array(n))
        dt = -math.log(u2) / total
        clock += dt
    return clock, dt


def _fixed(d, T, steps):
    dt = 1.0 / max(1e13 * math.exp(-float(x['Em_eV']) / (KB * T)) for x in d if int(x['mobility']) != wl.IMMOBILE)
    clock = 0.0
    for _ in range(steps):
        clock += dt
    return clock, dt


def _stats(clock, dt):
    return {'events': None, 'steps': None, 'solves': None, 'negative_barriers': None, 'clock': clock, 'dt_last': dt}


def exact(case, seed):
    do, n, C = case['do'], None if case['do'] == 'batch' else _dims(case), _constants(case)
    if do == 'batch':
        got = [_stats(*_residence(d, m, T, case['steps'], seed, C)) for m, d, T in _replicas(case, seed)]
        return {'positions': [None] * len(got), 'stats': got}
    d = _defects(case, seed)
    if do == 'kinetics':
        return {'positions': None, 'stats': _stats(*_fixed(d, 300.0, case['steps']))}
    if do == 'step':
        t = _fixed(d, case['T'], case['steps']) if case['fixed'] else _residence(d, n, case['T'], case['steps'], seed, C)
        return {'positions': None, 'stats': _stats(*t)}
    if do == 'static':
        return {'stress': _solve(_field(d, d['pos'], n).float().double(), n, C)}
    if do == 'setup':
        W = _SelfTerms(n, C)
        return {'self_terms': torch.stack([W.table(x) for x in d])}
    if do == 'shift':
        return {'energies': _shift(d, n, C, d['pos'][0] * (0.5 * H) + _shift_points(case, seed))}
    pos = _moved(d, n, 0 if do == 'solve' else case.get('moved', 1), seed).astype(np.int64)
    if do == 'solve':
        return {'stress': _solve(_field(d, pos, n), n, C)}
    if do == 'profile':
        sig = _solve(_field(d, pos, n), n, C)
        dip = np.array([_dipole(d, pos, i, sig, n, C) for i in range(len(d))])
        return {'site': _energies(d, pos, n, C, _SelfTerms(n, C), False, sig)[0], 'dipole': dip[:, 0], 'dipole_jumps': dip[:, 1:]}
    site, jumps = _energies(d, pos, n, C, _SelfTerms(n, C))
    return {'site': site, 'jumps': jumps}


def _dipole(d, pos, i, sig, n, C):
    """-(int eps*) : stress of the others at the centre of the site and of its eight jumps."""
    sig = sig - _solve(_field(d[i:i + 1], pos[i:i + 1], n), n, C)
    out = []
    for Y in [pos[i]] + [pos[i] + j for j in _JUMPS]:
        corner = [np.zeros(3, int)] if Y[0] & 1 else [-np.array([a, b, c]) for a in (0, 1) for b in (0, 1) for c in (0, 1)]
        v = _voxels(torch.tensor(np.array(corner), device='cuda'), np.asarray(Y) // 2, n)
        _, w, e = _stencil(d[i], 0)
        out.append(float(-KAPPA * H ** 3 * w.sum() * ((e * _DOUBLE.cuda()) @ sig.view(6, -1)[:, v].mean(dim=1))))
    return out


def _shift(d, n, C, X):
    """kappa int sigma(others) : (elastic strain of defect 0 moved to X), by Parseval."""
    rest = torch.fft.fftn(_solve(_field(d[1:], d['pos'][1:], n), n, C), dim=(1, 2, 3))
    own = torch.fft.fftn(_solve(_field(d[:1], np.zeros((1, 3), int), n), n, C), dim=(1, 2, 3))
    den = (C[0] - C[1]) * (C[0] + 2 * C[1])
    s11, s12 = (C[0] + C[1]) / den, -C[1] / den
    tr = own[0] + own[1] + own[2]
    A = sum(rest[a].conj() * ((s11 - s12) * own[a] + s12 * tr) for a in range(3))
    A = A + sum(rest[a].conj() * own[a] / C[2] for a in (3, 4, 5))
    f = [torch.fft.fftfreq(k, dtype=torch.float64, device='cuda') for k in n]
    E = []
    for x in X:
        ph = [torch.exp(-2j * math.pi * f[a] * (float(x[a]) / H)) for a in range(3)]
        E.append(float(((A * ph[0]).sum(-1) * ph[1]).sum(-1).mul(ph[2]).sum().real))
    return np.array(E) * KAPPA * H ** 3 / (n[0] * n[1] * n[2])
