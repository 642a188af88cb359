"""The work a user of this framework has it do, as measurable cases.

Every case goes through a public entry point of the package:

* ``point``: one energy / force / virial evaluation from host arrays (``DPA1.compute``);
* ``relax``: energy with coordinate and box gradients through ``autograd.energy`` in
  single precision, as a geometry or cell optimiser written in PyTorch calls it;
* ``box``: one evaluation on device arrays (``DPA1.compute_device``), the call of an MD engine;
* ``slab``: the same for one sub-domain with ghost atoms (``nlocal``), the call of one rank of a
  domain-decomposed engine;
* ``md``: velocity-Verlet steps replayed from one CUDA graph (``md.run``), continued from a
  saved state, with the full model or with the distilled student;
* ``batch``: uneven frames from host arrays in one call (``DPA1.compute_batch``);
* ``train``: the gradient of one batch of the student's training
  (``zero_grad``, ``train_frame``, ``get_grad``).

The systems are the seeded protein-like boxes and the water box of ``synth``; the models are its
default model (strip and concat type embedding), the model of the paper's size and the student.
"""

from __future__ import annotations

import dataclasses
import math
import os
import tempfile

import numpy as np
import torch

import synth
import paper_2604_07276_gb300 as dp
from paper_2604_07276_gb300 import autograd as dp_autograd
from paper_2604_07276_gb300 import md as dp_md

MODELS = {
    "default": synth.DEFAULT_CONFIG,
    "concat": dataclasses.replace(synth.DEFAULT_CONFIG, tebd_input_mode="concat"),
    "paper": synth.PAPER_SIZE_CONFIG,
    "student": synth.STUDENT_CONFIG,
}
ACC = 9.648533212e-3  # A / fs^2 per eV / (A amu)


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # the smallest call: single point of a 192-atom water box, from and to host memory
        {"name": "point_192", "kind": "point", "model": "default", "precision": "fp16x", "natoms": 192, "water": True},
        # one optimiser step of a small solvated peptide (single precision, cell gradient, the
        # original type-embedding form)
        {"name": "relax_582_concat", "kind": "relax", "model": "concat", "precision": "fp16x", "natoms": 582,
         "density": 0.1},
        # MD of a small protein: what a graph-replayed inner loop of ten steps costs
        {"name": "md_582", "kind": "md", "model": "default", "precision": "fp16x", "natoms": 582, "density": 0.1,
         "steps": 10},
        # the headline: one force evaluation of the 15,668-atom solvated protein
        {"name": "box_15668", "kind": "box", "model": "default", "precision": "fp16x", "natoms": 15668, "density": 0.1},
        # the same box with BF16 operands in two terms
        {"name": "box_15668_bf16x", "kind": "box", "model": "default", "precision": "bf16x", "natoms": 15668,
         "density": 0.1},
        # the single-precision path, as used to check the 16-bit ones
        {"name": "box_3001_fp32", "kind": "box", "model": "default", "precision": "fp32", "natoms": 3001,
         "density": 0.1},
        # one of four ranks of a domain-decomposed run of the 15,668-atom box: local atoms plus halo
        {"name": "slab_15668_of_4", "kind": "slab", "model": "default", "precision": "fp16x", "natoms": 15668,
         "density": 0.1, "slabs": 4},
        # the model of the paper's size on a mid-sized box
        {"name": "paper_3001_bf16x", "kind": "box", "model": "paper", "precision": "bf16x", "natoms": 3001,
         "density": 0.1},
        # labelling a data set: 32 uneven frames from host memory in one call
        {"name": "batch_32", "kind": "batch", "model": "default", "precision": "fp16x", "frames": 32, "lo": 200,
         "hi": 3000, "density": 0.1},
        # one training batch of the distilled student
        {"name": "train_16x582", "kind": "train", "model": "student", "precision": "bf16x", "frames": 16,
         "natoms": 582, "density": 0.1},
        # the student's MD between two checks by the full model
        {"name": "student_md_15668", "kind": "md", "model": "student", "precision": "fp16x", "natoms": 15668,
         "density": 0.1, "steps": 10},
        # a large box in one call
        {"name": "box_100003", "kind": "box", "model": "default", "precision": "fp16x", "natoms": 100003,
         "density": 0.1},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _density(rng, natoms):
    # from a dilute solution to a packed box; the box edge has to exceed twice the cutoff
    return round(min(rng.uniform(0.03, 0.12), natoms / 1950.0), 4)


# largest drawn box per model and precision: about the time of the largest listed case
_BOX_MAX = {("default", "fp16x"): 90000, ("concat", "fp16x"): 90000, ("default", "bf16x"): 30000,
            ("concat", "bf16x"): 30000, ("default", "fp32"): 10000, ("concat", "fp32"): 10000,
            ("paper", "bf16x"): 14000, ("paper", "fp32"): 4000}


def draw(rng):
    kind = rng.choice(["point", "relax", "md", "box", "box", "slab", "batch", "train", "student_md"])
    model, precision = rng.choice(sorted(_BOX_MAX))
    if kind == "point":
        n = _log(rng, 192, 3000)
        return {"kind": "point", "model": model, "precision": precision, "natoms": n, "density": _density(rng, n)}
    if kind == "relax":
        n = _log(rng, 192, 3000)
        return {"kind": "relax", "model": model, "precision": precision, "natoms": n, "density": _density(rng, n)}
    if kind == "md":
        n = _log(rng, 192, 4000)
        return {"kind": "md", "model": "default", "precision": "fp16x", "natoms": n, "density": _density(rng, n),
                "steps": 10}
    if kind == "box":
        n = _log(rng, 500, _BOX_MAX[model, precision])
        return {"kind": "box", "model": model, "precision": precision, "natoms": n, "density": _density(rng, n)}
    if kind == "slab":
        n = _log(rng, 4000, 40000)
        precision = rng.choice(["fp16x", "bf16x"])
        return {"kind": "slab", "model": "default", "precision": precision, "natoms": n,
                "density": round(rng.uniform(0.06, 0.11), 4), "slabs": rng.randint(2, 6)}
    if kind == "batch":
        lo = _log(rng, 200, 800)
        return {"kind": "batch", "model": rng.choice(["default", "concat"]), "precision": "fp16x",
                "frames": rng.randint(3, 40), "lo": lo, "hi": lo + rng.randint(50, 2000), "density": 0.1}
    if kind == "train":
        n = _log(rng, 192, 8000)
        return {"kind": "train", "model": "student", "precision": rng.choice(["bf16x", "fp32"]),
                "frames": max(1, min(16, 16000 // n)), "natoms": n, "density": _density(rng, n)}
    n = _log(rng, 582, 12000)
    return {"kind": "md", "model": "student", "precision": rng.choice(["fp16x", "bf16x", "fp32"]), "natoms": n,
            "density": _density(rng, n), "steps": 10}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _weights(case):
    """(config, weights) of the case's model."""
    if case["model"] == "student":
        # the student of the distillation set-up, 3 % off its teacher's base in training
        cfg, w = synth.teacher_base_weights(synth.TEACHER_BASE_OUT_SCALE)
        return cfg, synth.perturbed(w, 0.03, seed=7) if case["kind"] == "train" else w
    cfg = MODELS[case["model"]]
    return cfg, synth.make_weights(cfg, seed=0)


def _model(case):
    cfg, w = _weights(case)
    with tempfile.TemporaryDirectory() as d:
        path = os.path.join(d, "w.bin")
        synth.write_weights(path, cfg, w)
        return dp.DPA1(path, precision=case["precision"], device=0)


def _system(case, seed):
    if case.get("water"):
        return synth.water_box(seed=seed)
    return synth.lattice_system(case["natoms"], seed=seed, density=case["density"])


def _slab(case, seed):
    """(coord, atype, box, nlocal): an equal share of the box's atoms along x, then the halo atoms of
    either face (a quarter more than lie within rcut on average), as explicit copies in a box that
    keeps y and z periodic and leaves nothing within reach along x."""
    coord, atype, box = _system(case, seed)
    n, L, rcut = len(atype), float(box[0]), MODELS[case["model"]].rcut
    order = np.argsort(coord[:, 0], kind="stable")
    nlocal, halo = n // case["slabs"], int(1.25 * n * rcut / L)
    rows = np.concatenate([order[:nlocal], order[n - halo:], order[nlocal:nlocal + halo]])
    x = coord[rows].copy()
    x[nlocal:nlocal + halo, 0] -= L
    x[:, 0] += 3.0 * rcut
    return x, atype[rows], np.array([2.0 * L + 6.0 * rcut, box[1], box[2]]), nlocal


def _batch(case, seed):
    sizes = np.linspace(case["lo"], case["hi"], case["frames"]).round().astype(int)
    return [synth.lattice_system(int(n), seed=seed * 64 + k, density=case["density"])
            for k, n in enumerate(np.random.default_rng(3).permutation(sizes))]


def _train_frames(case, seed):
    """Frames with the energies and forces of the teacher's base."""
    cfg, w = synth.teacher_base_weights(synth.TEACHER_BASE_OUT_SCALE)
    ref = _Reference(cfg, w)
    out = []
    for k in range(case["frames"]):
        coord, atype, box = synth.lattice_system(case["natoms"], seed=seed * 64 + k, density=case["density"])
        e, f, _, _ = ref.evaluate(coord, box, atype)
        out.append((coord, atype, box, float(e), f))
    return out


def _velocities(case, atype, seed):
    # seeded weights have no short-range repulsion: trajectories are kept cold and short
    return synth.maxwell_boltzmann(atype, 10.0, seed=seed)


def _dt(case):
    # the full model's forces change faster than the student's
    return 0.25 if case["model"] == "student" else 0.1


def _dev(a, dtype):
    return torch.tensor(np.asarray(a), dtype=dtype, device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "model": _model(case)}
    if kind == "point":
        s["coord"], s["atype"], s["box"] = _system(case, seed)
        s["model"].reserve(len(s["atype"]))
    elif kind == "relax":
        coord, atype, box = _system(case, seed)
        s["coord"] = _dev(coord, torch.float32).requires_grad_()
        s["box"] = _dev(dp.box9(box), torch.float32).requires_grad_()
        s["atype"] = _dev(atype, torch.int32)
        s["model"].reserve(len(atype))
    elif kind in ("box", "slab"):
        if kind == "slab":
            coord, atype, box, s["nlocal"] = _slab(case, seed)
        else:
            (coord, atype, box), s["nlocal"] = _system(case, seed), None
        n = len(atype)
        s["coord"], s["atype"] = _dev(coord, torch.float64), _dev(atype, torch.int32)
        s["box"] = _dev(dp.box9(box), torch.float64)
        s["energy"] = torch.zeros(1, dtype=torch.float64, device="cuda")
        s["force"] = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
        s["virial"] = torch.zeros(9, dtype=torch.float64, device="cuda")
        s["atom_energy"] = torch.zeros(n, dtype=torch.float64, device="cuda")
        s["model"].reserve(n)
    elif kind == "md":
        coord, atype, box = _system(case, seed)
        vel = _velocities(case, atype, seed)
        s["md"] = dp_md.MDState(coord, vel, synth.MASSES[atype], box, atype)
        s["coord"], s["vel"] = s["md"].coord.clone(), s["md"].vel.clone()
        s["dt"], s["steps"] = _dt(case), case["steps"]
        s["model"].reserve(len(atype))
    elif kind == "batch":
        s["frames"] = _batch(case, seed)
    else:
        s["frames"] = [(_dev(c, torch.float64), _dev(dp.box9(b), torch.float64), _dev(t, torch.int32), e,
                        _dev(f, torch.float64)) for c, t, b, e, f in _train_frames(case, seed)]
        s["loss"] = torch.zeros((len(s["frames"]), 3), dtype=torch.float64, device="cuda")
        s["model"].reserve(case["natoms"])
    return s


def run(s):
    kind, m = s["kind"], s["model"]
    if kind == "point":
        e, f, w, ae = m.compute(s["coord"], s["box"], s["atype"], atom_energy=True)
        return {"energy": e, "force": f, "virial": w, "atom_energy": ae}
    if kind == "relax":
        e = dp_autograd.energy(s["coord"], m, s["box"], s["atype"])
        g_coord, g_box = torch.autograd.grad(e, (s["coord"], s["box"]))
        return {"energy": e.detach(), "g_coord": g_coord, "g_box": g_box}
    if kind in ("box", "slab"):
        m.compute_device(s["coord"], s["box"], s["atype"], s["energy"], s["force"], s["virial"], s["atom_energy"],
                         nlocal=s["nlocal"])
        return {k: s[k] for k in ("energy", "force", "virial", "atom_energy")}
    if kind == "md":
        md = s["md"]
        md.coord.copy_(s["coord"])  # back to the saved state
        md.vel.copy_(s["vel"])
        thermo = dp_md.run(m, md, dt=s["dt"], nsteps=s["steps"], graph=True)
        return {"coord": md.coord, "vel": md.vel, "force": md.force, "thermo": thermo}
    if kind == "batch":
        e, f, w = m.compute_batch(s["frames"])
        return {"energy": e, "force": np.concatenate(f), "virial": w}
    st = torch.cuda.current_stream().cuda_stream
    m.zero_grad(stream=st)
    for k, (coord, box, atype, e_ref, f_ref) in enumerate(s["frames"]):
        m.train_frame(coord, box, atype, e_ref, f_ref, s["loss"][k], stream=st)
    return {"grad": m.get_grad(), "loss": s["loss"]}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _model_flops(cfg, natoms, density):
    """Flops of one energy and force evaluation: every product of the network once forward and its
    adjoint once, over the neighbours that there are."""
    n = min(float(cfg.sel), max(1.0, density * 4.0 / 3.0 * math.pi * cfg.rcut ** 3))
    e0, e1, m1 = cfg.embed
    a = cfg.attn_dim
    embed = n * (e0 + e0 * e1 + e1 * m1)
    fwd = n * (2 * a * m1 + m1 * m1) + n * n * (a + m1)   # [Q K], output product; S, P G
    bwd = n * (2 * a * m1 + m1 * m1) + n * n * (2 * a + 2 * m1)
    desc = 4 * m1 * n + 4 * m1 * cfg.axis
    fit, fan = 0, cfg.fit_in
    for w in cfg.fitting:
        fit, fan = fit + fan * w, w
    mac = 2 * embed + cfg.attn_layers * (fwd + bwd) + 3 * desc + 2 * (fit + fan)
    return 2.0 * mac * natoms


def _model_bytes(cfg, natoms):
    """Coordinates, types and weights in; forces and atomic energies out."""
    weights = sum(int(np.prod(shape)) for _, shape in synth.model.tensor_order(cfg))
    return natoms * (24 + 4 + 24 + 8) + 4 * weights


def work(case):
    cfg, kind = MODELS[case["model"]], case["kind"]
    n, density = case.get("natoms", 0), case.get("density", 0.1)
    if kind == "batch":
        n = case["frames"] * (case["lo"] + case["hi"]) / 2
    if kind == "slab":  # the local atoms are the centres; the ghosts are read and get forces
        edge = (n / density) ** (1.0 / 3.0)
        local = n / case["slabs"]
        return {"bytes": _model_bytes(cfg, local + 2.5 * cfg.rcut * n / edge),
                "flops": _model_flops(cfg, local, density)}
    passes = 1
    if kind == "md":
        passes = case["steps"] + 1
    elif kind == "train":  # the evaluation and its tangent, each with its weight gradients
        return {"bytes": case["frames"] * _model_bytes(cfg, n), "flops": 4.0 * case["frames"] * _model_flops(cfg, n, density)}
    return {"bytes": passes * _model_bytes(cfg, n), "flops": passes * _model_flops(cfg, n, density)}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

class _Reference:
    """The model as plain FP64 tensor operations; derivatives by reverse mode."""

    def __init__(self, cfg, weights):
        self.cfg = cfg
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.t = {k: torch.tensor(np.asarray(v), dtype=torch.float64, device=self.dev) for k, v in weights.items()}

    def _net(self, x, prefix, layers):
        for l in range(layers):
            W, b = self.t[f"{prefix}_W{l}"], self.t[f"{prefix}_b{l}"]
            y = torch.tanh(x @ W + b)
            if W.shape[1] == W.shape[0]:
                y = x + y
            elif W.shape[1] == 2 * W.shape[0]:
                y = torch.cat([x, x], dim=-1) + y
            x = y
        return x

    def neighbours(self, x, L, centres):
        """([C, sel] ids padded with -1) the nearest sel atoms within rcut, by distance and index."""
        out = []
        rc2, n = self.cfg.rcut ** 2, x.shape[0]
        ids = torch.arange(n, device=self.dev)
        for c in centres.split(max(1, (1 << 24) // max(n, 1))):
            d = x[None, :, :] - x[c][:, None, :]
            d = d - L * torch.round(d / L)
            d2 = (d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1]) + d[..., 2] * d[..., 2]
            d2 = torch.where((d2 < rc2) & (ids[None, :] != c[:, None]), d2, torch.full_like(d2, math.inf))
            v, j = torch.topk(d2, min(self.cfg.sel, n), dim=1, largest=False, sorted=True)
            j = torch.where(torch.isfinite(v), j, torch.full_like(j, -1))
            out.append(torch.nn.functional.pad(j, (0, self.cfg.sel - j.shape[1]), value=-1))
        return torch.cat(out)

    def atomic_energies(self, rij, nlist, tc, tn):
        cfg, t = self.cfg, self.t
        mask = (nlist >= 0).to(torch.float64)
        r = torch.sqrt((rij * rij).sum(-1))
        u = (r - cfg.rcut_smth) / (cfg.rcut - cfg.rcut_smth)
        w = torch.where(r < cfg.rcut_smth, torch.ones_like(r), u ** 3 * (-6.0 * u * u + 15.0 * u - 10.0) + 1.0)
        w = w * mask
        s, rhat = w / r, rij / r[..., None] * mask[..., None]
        R = torch.cat([s[..., None], s[..., None] * rhat], dim=-1)
        R = (R - t["davg"][tc][:, None]) / t["dstd"][tc][:, None] * mask[..., None]
        Z = torch.tanh(t["te_W"] + t["te_b"])
        if cfg.tebd_input_mode == "concat":
            zj, zi = Z[tn], Z[tc][:, None].expand(*tn.shape, Z.shape[1])
            G = self._net(torch.cat([R[..., :1], zj, zi], dim=-1), "em", len(cfg.embed))
        else:
            nt = Z.shape[0]
            pair = torch.cat([Z[None, :].expand(nt, nt, -1), Z[:, None].expand(nt, nt, -1)], dim=-1)
            Gt = self._net(pair, "tt", len(cfg.embed))
            G = self._net(R[..., :1], "em", len(cfg.embed)) * (1.0 + Gt[tc[:, None], tn])
        G = G * mask[..., None]
        ww, gate = w[:, :, None] * w[:, None, :], rhat @ rhat.transpose(1, 2)
        for l in range(cfg.attn_layers):
            p = {k: t[f"at{l}_{k}"] for k in ("Wq", "bq", "Wk", "bk", "Wv", "bv", "Wo", "bo", "ln_g", "ln_b")}
            q, k, v = G @ p["Wq"] + p["bq"], G @ p["Wk"] + p["bk"], G @ p["Wv"] + p["bv"]
            logit = (q @ k.transpose(1, 2) / math.sqrt(cfg.attn_dim) + cfg.attn_shift) * ww - cfg.attn_shift
            att = torch.softmax(logit.masked_fill(mask[:, None, :] == 0, -1e30), dim=-1)
            y = (att * ww * gate) @ v @ p["Wo"] + p["bo"]
            y = y - y.mean(-1, keepdim=True)
            y = y / torch.sqrt((y * y).mean(-1, keepdim=True) + cfg.ln_eps)
            G = G + (y * p["ln_g"] + p["ln_b"]) * mask[..., None]
        T = R.transpose(1, 2) @ G / cfg.sel
        D = T.transpose(1, 2) @ T[:, :, :cfg.axis]
        h = self._net(torch.cat([D.reshape(D.shape[0], -1), Z[tc]], dim=-1), "fit", len(cfg.fitting))
        nf = len(cfg.fitting)
        return t["out_scale"] * (h @ t[f"fit_W{nf}"] + t[f"fit_b{nf}"])[:, 0] + t["ebias"][tc]

    def _inputs(self, coord, box, atype):
        x = torch.as_tensor(np.asarray(coord, dtype=np.float64), device=self.dev).clone()
        b = np.asarray(box, dtype=np.float64)
        h = torch.as_tensor(np.diag(b) if b.shape == (3,) else b.reshape(3, 3), device=self.dev).clone()
        return x, h, torch.as_tensor(np.asarray(atype, dtype=np.int64), device=self.dev)

    def _rows(self, x, h, atype, c, nl):
        """Displacement rows of centres c (padding rows (1, 0, 0)) and the neighbours' types."""
        j = nl.clamp(min=0)
        d = x[j] - x[c][:, None, :]
        image = -torch.round(d.detach() / torch.diagonal(h).detach())
        rij = d + image @ h
        pad = torch.zeros_like(rij)
        pad[..., 0] = 1.0
        return torch.where((nl >= 0)[..., None], rij, pad), atype[j]

    def evaluate(self, coord, box, atype, nlocal=None):
        """(E, F, dE/dh, (W, e)) as numpy arrays."""
        x, h, t = self._inputs(coord, box, atype)
        x.requires_grad_()
        h.requires_grad_()
        n = x.shape[0]
        nlocal = n if nlocal is None else nlocal
        e_all = torch.zeros(n, dtype=torch.float64, device=self.dev)
        W = torch.zeros(3, 3, dtype=torch.float64, device=self.dev)
        chunk = 512 if self.cfg.attn_layers else 4096
        L = torch.diagonal(h).detach()
        for c in torch.arange(nlocal, device=self.dev).split(chunk):
            nl = self.neighbours(x.detach(), L, c)
            rij, tn = self._rows(x, h, t, c, nl)
            rij.retain_grad()
            e = self.atomic_energies(rij, nl, t[c], tn)
            e.sum().backward()
            e_all[c] = e.detach()
            W -= (rij.detach() * (nl >= 0)[..., None]).reshape(-1, 3).T @ rij.grad.reshape(-1, 3)
        return (e_all.sum().item(), -x.grad.cpu().numpy(), h.grad.cpu().numpy(),
                (W.cpu().numpy(), e_all.cpu().numpy()))

    def loss_gradient(self, names, coord, box, atype, e_ref, f_ref):
        """((L, L_E, L_F), dL/dtheta) of one training frame."""
        leaves = [self.t[k].detach().clone().requires_grad_() for k in names]
        self.t.update(zip(names, leaves))
        x, h, t = self._inputs(coord, box, atype)
        x.requires_grad_()
        n = x.shape[0]
        c = torch.arange(n, device=self.dev)
        nl = self.neighbours(x.detach(), torch.diagonal(h), c)
        # forces chunk by chunk, then the loss's weight gradient with v = F - F_ref held:
        # dL/dtheta = 2 (E - E_ref) / N^2 dE/dtheta - 2 / (3 N) d(sum v . dE/dx)/dtheta
        E, f = 0.0, torch.zeros_like(x)
        for ci in c.split(1024):
            rij, tn = self._rows(x, h, t, ci, nl[ci])
            e = self.atomic_energies(rij, nl[ci], t[ci], tn).sum()
            f -= torch.autograd.grad(e, x)[0]
            E += e.item()
        v = f - torch.as_tensor(np.asarray(f_ref), device=self.dev)
        total = [torch.zeros_like(p) for p in leaves]
        for ci in c.split(1024):
            rij, tn = self._rows(x, h, t, ci, nl[ci])
            e = self.atomic_energies(rij, nl[ci], t[ci], tn).sum()
            gx = torch.autograd.grad(e, x, create_graph=True)[0]
            obj = 2.0 * (E - e_ref) / n ** 2 * e - 2.0 / (3 * n) * (v * gx).sum()
            for acc, g in zip(total, torch.autograd.grad(obj, leaves)):
                acc += g
        l_e, l_f = ((E - e_ref) / n) ** 2, (v * v).mean().item()
        return (l_e + l_f, l_e, l_f), np.concatenate([g.cpu().numpy().ravel() for g in total])


def exact(case, seed):
    if work(case)["flops"] > 3e12:  # more than about 20 seconds
        return None
    kind = case["kind"]
    cfg, weights = _weights(case)
    ref = _Reference(cfg, weights)
    if kind == "point":
        coord, atype, box = _system(case, seed)
        e, f, _, (v, ae) = ref.evaluate(coord, box, atype)
        return {"energy": e, "force": f, "virial": v, "atom_energy": ae}
    if kind == "relax":
        coord, atype, box = _system(case, seed)
        coord = coord.astype(np.float32).astype(np.float64)
        box = np.asarray(box).astype(np.float32).astype(np.float64)
        e, f, gh, _ = ref.evaluate(coord, box, atype)
        return {"energy": e, "g_coord": -f, "g_box": gh.reshape(9)}
    if kind in ("box", "slab"):
        if kind == "slab":
            coord, atype, box, nlocal = _slab(case, seed)
        else:
            (coord, atype, box), nlocal = _system(case, seed), None
        e, f, _, (v, ae) = ref.evaluate(coord, box, atype, nlocal)
        return {"energy": np.array([e]), "force": f, "virial": v.reshape(9), "atom_energy": ae}
    if kind == "md":
        coord, atype, box = _system(case, seed)
        x, v, dt = coord.copy(), _velocities(case, atype, seed), _dt(case)
        mass = synth.MASSES[atype][:, None]
        e, f, _, _ = ref.evaluate(x, box, atype)
        thermo = []
        for _ in range(case["steps"]):
            v = v + 0.5 * dt * ACC * f / mass
            x = x + dt * v
            e, f, _, _ = ref.evaluate(x, box, atype)
            v = v + 0.5 * dt * ACC * f / mass
            ek = float(0.5 * (mass * v * v).sum() / ACC)
            thermo.append((e, ek, e + ek))
        return {"coord": x, "vel": v, "force": f, "thermo": np.array(thermo)}
    if kind == "batch":
        es, fs, vs = [], [], []
        for coord, atype, box in _batch(case, seed):
            e, f, _, (v, _) = ref.evaluate(coord, box, atype)
            es.append(e)
            fs.append(f)
            vs.append(v)
        return {"energy": np.array(es), "force": np.concatenate(fs), "virial": np.array(vs)}
    names = [f"em_{k}{l}" for l in range(len(cfg.embed)) for k in "Wb"]
    names += [f"fit_{k}{l}" for l in range(len(cfg.fitting) + 1) for k in "Wb"] + ["ebias"]
    grad, losses = 0.0, []
    for coord, atype, box, e_ref, f_ref in _train_frames(case, seed):
        loss, g = ref.loss_gradient(names, coord, box, atype, e_ref, f_ref)
        grad = grad + g
        losses.append(loss)
    return {"grad": grad, "loss": np.array(losses)}
