"""The work that programs have this library do, as cases that can be timed and checked.

A case names one call of the public binding (`kind`), the potential's order and
precision, and the atoms.  Every configuration is the BCC crystal of
paper_2011_12875_gb300.inputs with random displacements, a strain and, for the
ragged sizes, vacancies.

Mixed precision computes in float32 (relative error about 1e-7 to 1e-6) and
hands its results over in float64 buffers; a program that chose it keeps them in
float32, as `run` does here.  FP64 results stay float64.
"""
from __future__ import annotations

import math
from functools import lru_cache

import numpy as np
import torch

from paper_2011_12875_gb300 import autograd, inputs, snap

LARGEST_MD_FP64 = 2000      # atoms at 2J = 14
LARGEST_MD_MIXED = 16000    # atoms at 2J = 14


def listed():
    def case(name, kind, twojmax, mixed, **kw):
        c = {"name": name, "kind": kind, "twojmax": twojmax, "mixed": mixed, "cells": 10, "vacancies": 0,
             "configs": 1, "disp": 0.1, "strain": 0.0, "shuffled": False}
        c.update(kw)
        return c

    return [
        # one step of molecular dynamics on a small cell, double precision: latency and launches
        case("md_128_2j8_fp64", "md", 8, False, cells=4),
        # the paper's benchmark shape, mixed precision: the step of a production run
        case("md_2000_2j8_mixed", "md", 8, True),
        # the same run in double precision
        case("md_2000_2j8_fp64", "md", 8, False),
        # the high-order potential, both precisions
        case("md_2000_2j14_mixed", "md", 14, True),
        case("md_2000_2j14_fp64", "md", 14, False),
        # a large cell of the high-order potential
        case("md_16000_2j14_mixed", "md", 14, True, cells=20),
        # an engine that keeps its own neighbour list: ragged atom count, defects, atoms in no
        # spatial order, an order between the tuned ones
        case("list_1013_2j6_mixed", "list", 6, True, cells=8, vacancies=11, disp=0.2, shuffled=True),
        # an engine on the host: pinned positions in, energies and forces out, each step
        case("host_2000_2j8_mixed", "host", 8, True),
        # screening: 64 configurations of 54 to 2000 atoms at once
        case("batch_64_2j8_mixed", "batch", 8, True, configs=64, strain=0.02),
        # descriptors for an external model
        case("bispectrum_2000_2j8_mixed", "bispectrum", 8, True),
        # a fitting step (loss and gradient in the coefficients) over 32 configurations
        case("fit_32_2j8_mixed", "fit", 8, True, configs=32, disp=0.2),
        # energies inside a torch program, differentiated through autograd, double precision
        case("autograd_431_2j8_fp64", "autograd", 8, False, cells=6, vacancies=1, disp=0.15),
    ]


def draw(rng):
    kind = rng.choice(["md", "md", "md", "list", "host", "batch", "bispectrum", "fit", "autograd"])
    twojmax = rng.choice([2, 4, 5, 6, 7, 8, 8, 8, 10, 11, 12, 14, 14])
    mixed = rng.random() < 0.6
    several = kind in ("batch", "fit")
    # atoms: over the logarithm of 16 .. the most that costs no more than the largest listed case
    most = min(16000.0, (LARGEST_MD_MIXED if mixed else LARGEST_MD_FP64) * (14.0 / twojmax) ** (1 if mixed else 5))
    if kind in ("bispectrum", "fit"):
        most = min(most, 16000.0 if twojmax <= 8 else 2000.0) / (1 if mixed else 4)
    if several:
        sizes = _batch_sizes(kind)
        mean = 2.0 * sum(s ** 3 for s in sizes) / len(sizes)
        configs = max(2, min(64, int(math.exp(rng.uniform(math.log(2.0), math.log(max(2.1, most / mean)))))))
        cells, vacancies = 0, 0
    else:
        n = math.exp(rng.uniform(math.log(16.0), math.log(most)))
        cells, configs = max(2, min(20, round((n / 2.0) ** (1.0 / 3.0)))), 1
        atoms = 2 * cells ** 3
        vacancies = rng.randrange(0, max(1, atoms // 50) + 1) if rng.random() < 0.6 else 0
    return {"kind": kind, "twojmax": twojmax, "mixed": mixed, "cells": cells, "vacancies": vacancies,
            "configs": configs, "disp": round(rng.uniform(0.05, 0.2), 3), "strain": round(rng.uniform(0.0, 0.02), 4),
            "shuffled": rng.random() < 0.3}


# ------------------------------------------------------------------ inputs
def _batch_sizes(kind):
    return inputs.FIT_SIZES if kind == "fit" else inputs.BATCH_SIZES


def _configs(case, seed):
    """The case's configurations: positions and boxes in float64, on the host."""
    g = np.random.Generator(np.random.PCG64([seed, 17]))
    several = case["kind"] in ("batch", "fit")
    # the cells of a batch do not depend on the seed: the same work for every input
    pick = np.random.Generator(np.random.PCG64([case["configs"], case["twojmax"]]))
    cells = pick.choice(np.array(_batch_sizes(case["kind"])), size=case["configs"]) if several else [case["cells"]]
    out = []
    for nc in cells:
        c = inputs.bcc(int(nc), disp=case["disp"], strain=case["strain"], seed=int(g.integers(1 << 31)))
        pos = c.pos
        if case["vacancies"]:
            keep = np.sort(g.permutation(len(pos))[case["vacancies"]:])
            pos = pos[keep]
        if case["shuffled"]:
            pos = pos[g.permutation(len(pos))]
        out.append((np.ascontiguousarray(pos), c.box))
    return out


def _beta(case, seed):
    return inputs.beta(case["twojmax"], seed=seed + 5)


def _forces_ref(case, n, seed):
    return np.random.Generator(np.random.PCG64([seed, 23])).normal(scale=0.5, size=(n, 3))


def _weights(case, n, seed):
    return np.random.Generator(np.random.PCG64([seed, 29])).uniform(0.5, 1.5, size=n)


def _natoms(case):
    if case["kind"] in ("batch", "fit"):
        return sum(len(p) for p, _ in _configs(case, 0))
    return 2 * case["cells"] ** 3 - case["vacancies"]


def prepare(case, seed):
    dev = torch.device("cuda:0")
    cfgs = _configs(case, seed)
    pos = np.concatenate([p for p, _ in cfgs])
    n, kind, mixed = len(pos), case["kind"], case["mixed"]
    st = {"kind": kind, "mixed": mixed, "box": cfgs[0][1],
          "model": snap.Snap(case["twojmax"], _beta(case, seed), precision=snap.MIXED if mixed else snap.FP64)}
    if kind == "host":
        def pinned(shape):
            return torch.empty(shape, dtype=torch.float64, pin_memory=True).numpy()

        st["pos"] = pinned((n, 3))
        st["pos"][:] = pos
        st["out"] = (pinned((n,)), pinned((n, 3)), pinned((6,)))
        return st
    st["pos"] = torch.tensor(pos, dtype=torch.float64, device=dev)
    if kind in ("md", "list"):
        # the engine's own result arrays, one block
        buf = torch.empty(4 * n + 6, dtype=torch.float64, device=dev)
        st["buf"] = buf
        st["out"] = (buf[:n], buf[n:4 * n].view(n, 3), buf[4 * n:])
        st["single"] = torch.empty(4 * n + 6, dtype=torch.float32, device=dev) if mixed else None
    if kind == "list":
        st["list"] = _neighbour_list(st["pos"], cfgs[0][1], 40)
    if kind in ("batch", "fit"):
        st["natoms"] = np.array([len(p) for p, _ in cfgs], dtype=np.int32)
        st["boxes"] = np.array([b for _, b in cfgs])
    if kind == "fit":
        st["f_ref"] = torch.tensor(_forces_ref(case, n, seed), dtype=torch.float64, device=dev)
    if kind == "autograd":
        st["pos"].requires_grad_(True)
        st["w"] = torch.tensor(_weights(case, n, seed), dtype=torch.float64, device=dev)
    return st


def run(st):
    kind, model = st["kind"], st["model"]
    if kind in ("md", "list"):
        # steps are enqueued one after the other; a program looks at the errors now and then
        e, f, w = st["out"]
        model.compute(st["pos"], st["box"], energy=e, forces=f, virial=w, neighbors=st.get("list"), wait=False)
        if not st["mixed"]:
            return e, f, w
        single, n = st["single"], e.shape[0]
        single.copy_(st["buf"])
        return single[:n], single[n:4 * n].view(n, 3), single[4 * n:]
    if kind == "host":
        e, f, w = model.compute_host(st["pos"], st["box"], out=st["out"])
        return tuple(x.astype(np.float32) for x in (e, f, w)) if st["mixed"] else (e, f, w)
    if kind == "batch":
        out = model.compute_batch(st["pos"], st["natoms"], st["boxes"])
    elif kind == "bispectrum":
        out = (model.bispectrum(st["pos"], st["box"]),)
    elif kind == "fit":
        out = autograd.force_matching_grad_batch(model, st["pos"], st["natoms"], st["boxes"], st["f_ref"])
    else:
        e = autograd.energy(model, st["pos"], st["box"])
        (g,) = torch.autograd.grad((e * st["w"]).sum(), st["pos"])
        out = (e.detach(), g)
    return tuple(x.float() for x in out) if st["mixed"] else out


# ---------------------------------------------------------------- the work
def _triples(twojmax):
    """(t1, t2, t) with t2 <= t1 <= t <= 2J, the ranks of the bispectrum components."""
    return [(t1, t2, t) for t1 in range(twojmax + 1) for t2 in range(t1 + 1)
            for t in range(t1, min(twojmax, t1 + t2) + 1) if (t1 + t2 + t) % 2 == 0]


@lru_cache(maxsize=None)
def _couplings(twojmax):
    """Products u u conj(u) of all components, those equal by the inversion symmetry once."""
    total = 0
    for t1, t2, t in _triples(twojmax):
        n = sum(1 for m1 in range(-t1, t1 + 1, 2) for m2 in range(-t2, t2 + 1, 2) if abs(m1 + m2) <= t)
        total += (n * n + 1) // 2
    return total


def work(case):
    n, J, kind = _natoms(case), case["twojmax"], case["kind"]
    pairs = 26 * n
    half = sum((t + 1) * (t // 2 + 1) for t in range(J + 1))
    comps = len(_triples(J))
    # u of a pair: a complex element from the last layer (4 products) and its sum
    flops = pairs * half * 10.0
    moved = 24.0 * n
    if kind == "list":
        moved += n * 4.0 + 7.0 * pairs
    if kind == "bispectrum":
        return {"bytes": moved + 8.0 * n * comps, "flops": flops + n * 4.0 * _couplings(J)}
    # the adjoint (a coupling feeds its three elements) and dE/dr of a pair: value and two
    # complex derivatives
    flops += n * 8.0 * _couplings(J) + pairs * half * 12.0
    moved += 32.0 * n
    if kind == "fit":
        # the tangent of u and the product rule over the couplings
        flops += pairs * half * 16.0 + n * 12.0 * _couplings(J)
        moved += 24.0 * n + 8.0 * comps
    return {"bytes": moved, "flops": flops}


# -------------------------------------------------------------- 64-bit truth
# Energies, forces, virial, descriptors and the fitting gradient in plain torch, from the
# definitions: full matrices, the layer recursion, dense Clebsch-Gordan couplings, and
# torch's own differentiation.

def _pairs(pos, box):
    """(i, k, separation, image) of every pair within the cutoff."""
    dev, n = pos.device, pos.shape[0]
    L = torch.tensor(np.asarray(box), dtype=torch.float64, device=dev)
    r = inputs.RCUT
    axes = [[0] if float(x) > 2.0 * r + 0.2 else list(range(-(int(r / float(x)) + 1), int(r / float(x)) + 2)) for x in L]
    shifts = torch.tensor([(x, y, z) for x in axes[0] for y in axes[1] for z in axes[2]], dtype=torch.float64, device=dev)
    found = []
    step = max(1, int(2e7) // (n * len(shifts)))
    for a in range(0, n, step):
        d = pos[None, :, :] - pos[a:a + step, None, :]
        near = -torch.round(d / L)
        im = near[:, :, None, :] + shifts
        full = d[:, :, None, :] + im * L
        i, k, s = torch.nonzero((full * full).sum(-1) < r * r, as_tuple=True)
        sep, img = full[i, k, s], im[i, k, s]
        other = ~((i + a == k) & (img == 0).all(-1))
        found.append((i[other] + a, k[other], sep[other], img[other]))
    return tuple(torch.cat(x) for x in zip(*found))


def _neighbour_list(pos, box, cap):
    """(count, index, image) as an engine hands its list over."""
    n = pos.shape[0]
    i, k, _, img = _pairs(pos, box)
    cnt = torch.bincount(i, minlength=n)
    slot = torch.arange(len(i), device=pos.device) - (torch.cumsum(cnt, 0) - cnt)[i]
    idx = torch.zeros((n, cap), dtype=torch.int32, device=pos.device)
    image = torch.zeros((n, cap, 3), dtype=torch.int8, device=pos.device)
    idx[i, slot] = k.to(torch.int32)
    image[i, slot] = img.to(torch.int8)
    return cnt.to(torch.int32), idx, image


def _cg(t1, m1, t2, m2, t, m):
    """Clebsch-Gordan coefficient of doubled ranks and projections (Racah's sum)."""
    f = math.factorial
    a, b, c = (t1 + t2 - t) // 2, (t1 - m1) // 2, (t2 + m2) // 2
    d, e = (t - t2 + m1) // 2, (t - t1 - m2) // 2
    s = 0.0
    for k in range(max(0, -d, -e), min(a, b, c) + 1):
        s += (-1.0) ** k / (f(k) * f(a - k) * f(b - k) * f(c - k) * f(d + k) * f(e + k))
    tri = f(a) * f((t1 - t2 + t) // 2) * f((t2 - t1 + t) // 2) * (t + 1) / f((t1 + t2 + t) // 2 + 1)
    proj = f((t1 + m1) // 2) * f(b) * f(c) * f((t2 - m2) // 2) * f((t + m) // 2) * f((t - m) // 2)
    return s * math.sqrt(tri * proj)


@lru_cache(maxsize=None)
def _coupling(t1, t2, t):
    """[(t1+1)(t2+1), t+1]: the coefficients that couple two rows to rank t."""
    c = np.zeros(((t1 + 1) * (t2 + 1), t + 1))
    for x1 in range(t1 + 1):
        for x2 in range(t2 + 1):
            m1, m2 = 2 * x1 - t1, 2 * x2 - t2
            if abs(m1 + m2) <= t:
                c[x1 * (t2 + 1) + x2, (m1 + m2 + t) // 2] = _cg(t1, m1, t2, m2, t, m1 + m2)
    return c


def _u_pairs(J, d):
    """f_c u_t of every pair: a list over t of [P, t+1, t+1] complex."""
    span = inputs.RCUT - inputs.RMIN0
    r = torch.sqrt((d * d).sum(-1))
    th = inputs.RFAC0 * math.pi * (r - inputs.RMIN0) / span
    z0 = r / torch.tan(th)
    r0 = torch.sqrt(r * r + z0 * z0)
    a = torch.complex(z0, -d[:, 2]) / r0
    b = torch.complex(d[:, 1], -d[:, 0]) / r0
    fc = 0.5 * (torch.cos(math.pi * (r - inputs.RMIN0) / span) + 1.0)
    ca, cb = a.conj()[:, None, None], b.conj()[:, None, None]
    u = torch.ones((len(r), 1, 1), dtype=torch.complex128, device=d.device)
    out = [u * fc[:, None, None]]
    for t in range(1, J + 1):
        ma = torch.arange(t + 1, dtype=torch.float64, device=d.device)
        mb = torch.arange(t, dtype=torch.float64, device=d.device)
        up = torch.sqrt((t - ma[:t, None]) / (t - mb[None, :]))
        dn = torch.sqrt(ma[1:, None] / (t - mb[None, :]))
        left = torch.nn.functional.pad(ca * up * u, (0, 0, 0, 1)) - torch.nn.functional.pad(cb * dn * u, (0, 0, 1, 0))
        # the last column from u[t-ma][t-mb] = (-1)^(ma+mb) conj(u[ma][mb])
        sign = torch.tensor([(-1.0) ** (t + m) for m in range(t + 1)], dtype=torch.float64, device=d.device)
        last = sign[:, None] * left[:, :, :1].conj().flip(1)
        u = torch.cat([left, last], dim=2)
        out.append(u * fc[:, None, None])
    return out


def _u_atoms(J, d, i, n):
    """Ulisttot: the pairs' sum and the atom's own part."""
    out = []
    for t, u in enumerate(_u_pairs(J, d)):
        s = torch.zeros((n, t + 1, t + 1), dtype=torch.complex128, device=d.device).index_add(0, i, u)
        out.append(s + torch.eye(t + 1, dtype=torch.complex128, device=d.device))
    return out


def _b(U, t1, t2, t):
    """Re Z : conj(U_t) of one component for every atom."""
    c = torch.tensor(_coupling(t1, t2, t), dtype=torch.complex128, device=U[t].device)
    n = U[t].shape[0]
    # kron of the two matrices, rows (ma1, ma2), columns (mb1, mb2)
    k = (U[t1][:, :, None, :, None] * U[t2][:, None, :, None, :]).reshape(n, -1, (t1 + 1) * (t2 + 1))
    z = c.T @ (k @ c)
    return (z * U[t].conj()).real.sum((1, 2))


def _b_grad(U, comp, scale, want):
    """One component of every atom (scaled): its values, and its gradient added to U's .grad."""
    t1, t2, t = comp
    n, vals = U[0].shape[0], []
    step = max(1, int(1.5e8) // ((t1 + 1) * (t2 + 1)) ** 2)
    for a in range(0, n, step):
        part = [x[a:a + step] for x in U]
        b = _b(part, t1, t2, t)
        vals.append(b.detach())
        if want:
            (b * scale).sum().backward()
    return torch.cat(vals)


def _evaluate(J, beta, pos, box, want="all"):
    """Energies, forces, virial, per-pair dE_i/dr_ik and the pairs; with want="B" the components."""
    n = pos.shape[0]
    i, k, sep, _ = _pairs(pos, box)
    d = sep.clone().requires_grad_(True)
    U = _u_atoms(J, d, i, n)
    comps = _triples(J)
    leaf = [x.detach().requires_grad_(want != "B") for x in U]
    if want == "B":
        with torch.no_grad():
            return torch.stack([_b_grad(leaf, c, 1.0, False) for c in comps], dim=1)
    e = torch.full((n,), float(beta[0]), dtype=torch.float64, device=pos.device)
    for l, c in enumerate(comps):
        e += float(beta[1 + l]) * _b_grad(leaf, c, float(beta[1 + l]), True)
    torch.autograd.backward(U, [x.grad for x in leaf])
    g = d.grad
    f = torch.zeros_like(pos).index_add(0, i, g).index_add(0, k, -g)
    w = torch.stack([-(g[:, a] * sep[:, b]).sum() for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))])
    return e, f, w, g, (i, k, sep)


def _fit_gradient(J, pairs, n, g):
    """-sum_i dB_l(i) along the displacement field g, for every component."""
    i, k, sep = pairs
    U, dU = torch.func.jvp(lambda d: tuple(_u_atoms(J, d, i, n)), (sep,), (g[k] - g[i],))
    leaf = [x.detach().requires_grad_(True) for x in U]
    out = [0.0]
    for c in _triples(J):
        for x in leaf:
            x.grad = None
        _b_grad(leaf, c, 1.0, True)
        out.append(-sum(float((x.grad.conj() * y).real.sum()) for x, y in zip(leaf, dU) if x.grad is not None))
    return out


def exact(case, seed):
    J, kind = case["twojmax"], case["kind"]
    if _natoms(case) * float(_couplings(J)) * (3.0 if kind == "fit" else 1.0) > 6e9:
        return None
    dev = torch.device("cuda:0" if torch.cuda.is_available() else "cpu")
    beta = _beta(case, seed)
    cfgs = [(torch.tensor(p, dtype=torch.float64, device=dev), b) for p, b in _configs(case, seed)]
    if kind == "bispectrum":
        return (_evaluate(J, beta, *cfgs[0], want="B"),)
    if kind == "fit":
        ref = torch.tensor(_forces_ref(case, sum(len(p) for p, _ in cfgs), seed), dtype=torch.float64, device=dev)
        loss, grad, start = 0.0, np.zeros(len(beta)), 0
        for p, b in cfgs:
            _, f, _, _, pairs = _evaluate(J, beta, p, b)
            r = f - ref[start:start + len(p)]
            loss += float((r * r).sum())
            grad += np.array(_fit_gradient(J, pairs, len(p), 2.0 * r))
            start += len(p)
        return torch.tensor(loss, dtype=torch.float64), torch.tensor(grad, dtype=torch.float64)
    if kind == "autograd":
        p, b = cfgs[0]
        e, _, _, g, (i, k, _) = _evaluate(J, beta, p, b)
        w = torch.tensor(_weights(case, len(p), seed), dtype=torch.float64, device=dev)
        wg = w[i][:, None] * g
        return e, torch.zeros_like(p).index_add(0, k, wg).index_add(0, i, -wg)
    parts = [_evaluate(J, beta, p, b)[:3] for p, b in cfgs]
    if kind == "batch":
        return torch.cat([x[0] for x in parts]), torch.cat([x[1] for x in parts]), torch.stack([x[2] for x in parts])
    return parts[0]
