"""What a user of this library has it do, as measurable cases through its public entry
points: latent steps and rollouts, decodes with derivatives, dense reconstructions,
full-order solves and training steps.  Sizes are those of the repository's workloads
(``workloads/gen.py``), tests and benchmark; ``draw`` spreads over the same ranges.

Every case is a dict with a ``kind``:

* ``step``    crom_step (``steps`` = 0) or crom_rollout (``steps`` > 0) from the codes q0
* ``decode``  crom_decode / crom_decode_tc: the decoder and its derivatives at points
* ``recon``   crom_reconstruct: the field at every point for several codes
* ``fom``     crom_fom_step: the explicit full-order solver
* ``train``   crom_train_step and its gradients
"""
import math

import numpy as np
import torch

from paper_2206_02607_gb300 import crom
from workloads import gen

PREC = {"fp32": crom.CROM_PREC_FP32, "f16x2": crom.CROM_PREC_F16X2, "f16": crom.CROM_PREC_F16,
        "bf16": crom.CROM_PREC_BF16_MIXED}
OMEGA0 = 30.0
FOM_KIND = {"heat1d": crom.CROM_FOM_HEAT1D_DIRICHLET, "heat2d": crom.CROM_FOM_HEAT2D_NEUMANN,
            "heat2d_field": crom.CROM_FOM_HEAT2D_NEUMANN_FIELD, "advdiff": crom.CROM_FOM_ADVDIFF2D_PERIODIC,
            "advdiff_central": crom.CROM_FOM_ADVDIFF2D_PERIODIC_CENTRAL}


def _step(name, **kw):
    c = {"name": name, "kind": "step", "prec": "fp32", "act": "elu", "m": 2, "r": 8, "width": 128, "hidden": 5,
         "n_inst": 1, "lo": 200, "hi": 200, "gn": 2, "steps": 0, "pde": "heat", "coef_per_sample": False, "dt": 1e-5}
    c.update(kw)
    return c


def listed():
    return [
        # one step of the smallest problem (1D heat, 16 samples): a caller that steps one
        # instance at a time pays launches and latency
        _step("step_heat1d_fp32", m=1, r=3, width=64, hidden=4, lo=16, hi=16, gn=1),
        # the plain 2D problem (200 samples, 2 Gauss-Newton iterations), 100 steps of its
        # rollout as one graph: the ordinary single-instance use
        _step("rollout_heat2d_fp32", steps=100),
        # a SIREN decoder, which only the FP32 path serves: a batch of uneven instances
        _step("step_siren_fp32", act="siren", n_inst=64, lo=32, hi=512, dt=1e-6),
        # the batched step on the tensor cores: 1024 uneven instances
        _step("step_batch_f16x2", prec="f16x2", n_inst=1024, lo=32, hi=512),
        # the learned model's rollout step: 8 held-out trajectories of the periodic
        # advection-diffusion problem, 4096 integration samples each, r = 15
        _step("step_advdiff_f16", prec="f16", r=15, n_inst=8, lo=4096, hi=4096, pde="advdiff", dt=2.5e-4),
        # every derivative channel of the decoder on the 128 x 128 grid (building a latent
        # step of one's own, inspecting a trained field)
        {"name": "decode_fp32", "kind": "decode", "prec": "fp32", "act": "elu", "m": 2, "r": 8, "width": 128, "hidden": 5,
         "n_inst": 1, "n_pts": 128 * 128, "want": 31},
        # dense fields of 16 codes on the 1024 x 1024 grid, the accurate tensor-core form
        {"name": "recon_dense_f16x2", "kind": "recon", "prec": "f16x2", "act": "elu", "m": 2, "r": 8, "width": 128, "hidden": 5,
         "n_codes": 16, "side": 1024},
        # the fields of the 8 held-out trajectories on 256 x 256 with the learned decoder's
        # other shape (width 256, r = 16), which the FP32 path reconstructs
        {"name": "recon_w256_fp32", "kind": "recon", "prec": "fp32", "act": "elu", "m": 2, "r": 16, "width": 256, "hidden": 5,
         "n_codes": 8, "side": 256},
        # the reference solution of the 2D heat problem: a few 128 x 128 fields, 100 steps
        {"name": "fom_heat2d", "kind": "fom", "model": "heat2d", "n": 128, "batch": 8, "steps": 100},
        # training data of the learned model: 64 trajectories on 256 x 256, the 10 steps
        # between two snapshots
        {"name": "fom_advdiff", "kind": "fom", "model": "advdiff_central", "n": 256, "batch": 64, "steps": 10},
        # a training step of the learned model: 64 snapshots x 4096 points, width 256
        {"name": "train_bf16", "kind": "train", "prec": "bf16", "m": 2, "r": 16, "width": 256, "hidden": 5, "side": 256,
         "B": 64, "S": 4096},
        # the same at the trainer's default precision, on the 48 x 48 heat problem's shapes
        {"name": "train_fp32", "kind": "train", "prec": "fp32", "m": 2, "r": 8, "width": 128, "hidden": 5, "side": 48,
         "B": 32, "S": 1024},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step_tc", "step_tc", "decode", "recon", "fom", "fom", "train", "train"])
    if kind == "step":
        c = _step("")
        c.update(m=rng.choice([1, 2, 2]), width=rng.choice([32, 64, 96, 128, 128, 160, 256]), hidden=rng.randint(2, 5),
                 n_inst=_log(rng, 1, 64), gn=rng.randint(1, 2))
        c["r"] = rng.randint(2, 4) if c["m"] == 1 else rng.randint(3, 8)
        c["lo"] = _log(rng, 16, 120)
        c["hi"] = min(_log(rng, c["lo"], 512), 250 if c["m"] == 1 else 512)
        c["hi"] = max(c["hi"], c["lo"])
        c["coef_per_sample"] = rng.random() < 0.25
        if rng.random() < 0.25:
            c.update(act="siren", dt=1e-6)
        elif c["m"] == 2 and rng.random() < 0.25:
            c.update(pde="advdiff", dt=2.5e-4)
        if c["n_inst"] <= 8 and rng.random() < 0.5:
            c["steps"] = _log(rng, 2, 50)
    elif kind == "step_tc":
        c = _step("", prec=rng.choice(["f16x2", "f16x2", "f16"]))
        c.update(hidden=rng.randint(3, 5), r=rng.randint(4, 15), n_inst=_log(rng, 1, 1024), gn=2)
        c["lo"] = _log(rng, 32, 256)
        c["hi"] = min(4096, max(c["lo"], _log(rng, c["lo"], max(c["lo"] + 1, 250000 // c["n_inst"]))))
        c["coef_per_sample"] = rng.random() < 0.25
        if rng.random() < 0.4:
            c.update(pde="advdiff", dt=2.5e-4)
        if c["n_inst"] <= 64 and rng.random() < 0.5:
            c["steps"] = _log(rng, 2, 10)
    elif kind == "decode":
        c = {"kind": "decode", "prec": rng.choice(["fp32", "fp32", "f16x2", "f16"]), "act": "elu", "m": 2, "width": 128,
             "r": rng.randint(3, 12), "hidden": rng.randint(2, 5), "n_inst": _log(rng, 1, 64)}
        if c["prec"] == "fp32":
            c.update(width=rng.choice([64, 96, 128, 256]), act=rng.choice(["elu", "elu", "siren"]))
            c["want"] = rng.choice([1, 3, 9, 17, 25, 31])
        else:
            c["want"] = rng.choice([1, 9, 11, 25, 27])
        c["n_pts"] = max(c["n_inst"], _log(rng, 200, 30000 if c["prec"] == "fp32" else 270000))
    elif kind == "recon":
        c = {"kind": "recon", "prec": rng.choice(["fp32", "f16x2", "f16"]), "act": "elu", "m": 2, "width": 128,
             "r": rng.randint(3, 15), "hidden": rng.randint(2, 5), "n_codes": _log(rng, 1, 16), "side": _log(rng, 48, 1024)}
        if c["prec"] == "fp32":
            c.update(width=rng.choice([64, 128, 256]), act=rng.choice(["elu", "elu", "siren"]),
                     side=_log(rng, 48, 256), n_codes=_log(rng, 1, 8))
    elif kind == "fom":
        c = {"kind": "fom", "model": rng.choice(sorted(FOM_KIND)), "steps": _log(rng, 1, 100)}
        if c["model"] == "heat1d":
            c.update(n=rng.choice([101, 256, 257, 1024]), batch=_log(rng, 1, 512))
        else:
            c["n"] = rng.choice([48, 64, 97, 128, 128, 200, 256, 256])
            c["batch"] = _log(rng, 1, max(2, min(512, 8 * 10 ** 8 // (c["n"] ** 2 * c["steps"]))))
    else:
        c = {"kind": "train", "prec": rng.choice(["bf16", "bf16", "fp32"]), "m": 2, "r": rng.randint(3, 16),
             "width": rng.choice([64, 128, 256]), "hidden": rng.randint(3, 5), "side": rng.choice([48, 64, 100, 128]),
             "B": _log(rng, 4, 64)}
        c["S"] = _log(rng, 100, 4096 if c["prec"] == "bf16" else 1024)
    c.pop("name", None)
    return c


# ------------------------------------------------------------------ inputs


def _decoder(case, rng_seed):
    spec = gen.DecoderSpec(case["m"], case["r"], case["width"], case["hidden"])
    if case.get("act") == "siren":
        return spec, gen.siren_decoder(spec, rng_seed, OMEGA0)
    return spec, gen.xavier_decoder(spec, rng_seed, bias_std=0.05)


def _dev(a, dtype):
    return torch.as_tensor(np.ascontiguousarray(a)).to(device="cuda", dtype=dtype)


def _inputs(case, seed):
    """The arrays of a case on the host, from the seed alone (shared by prepare and exact)."""
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind in ("step", "decode", "recon"):
        spec, params = _decoder(case, int(rng.integers(1 << 30)))
        siren = case.get("act") == "siren"
    if kind == "step":
        n, m, r = case["n_inst"], case["m"], case["r"]
        sizes = rng.integers(case["lo"], case["hi"] + 1, size=n)
        d = {"params": params, "sizes": sizes, "s_off": gen.ragged_offsets(sizes), "vel": None}
        if case["pde"] == "advdiff":
            # cell centres and velocities of the learned workload, coordinates standardised
            ax, ay = gen.stream_function_faces(256, rng)
            cen, vel = gen.cell_centers_2d(256), gen.cell_velocity(ax, ay)
            s = float(cen[:, 0].std())
            cells = np.concatenate([rng.choice(256 * 256, size=int(k), replace=False) for k in sizes])
            d["samples"], d["vel"] = ((cen[cells] - 0.5) / s).astype(np.float32), (vel[cells] / s).astype(np.float32)
            coef = rng.uniform(1e-3, 1e-2, size=n) / s ** 2
        else:
            nodes = (gen.interior_nodes_1d if m == 1 else gen.interior_nodes_2d)
            d["samples"] = np.concatenate([nodes(256 if m == 1 else 128, int(k), rng) for k in sizes])
            coef = rng.uniform(0.5, 2.0, size=n)
        if siren:
            d["samples"] = (2.0 * d["samples"] - 1.0).astype(np.float32)
        d["alpha"] = coef.astype(np.float32)
        if case["coef_per_sample"]:  # piecewise constant over four strips, scaled per instance
            x01 = (d["samples"] - d["samples"].min()) / np.ptp(d["samples"])
            d["alpha"] = (gen.piecewise_nu(x01, [0.25, 1.0, 0.5, 0.75]) * np.repeat(coef, sizes)).astype(np.float32)
        d["q0"] = rng.standard_normal((n, r)) * (0.5 if siren else 1.0)
        return d
    if kind == "decode":
        n, k = case["n_pts"], case["n_inst"]
        cuts = np.sort(rng.choice(np.arange(1, n), size=k - 1, replace=False)) if k > 1 else np.zeros(0, np.int64)
        off = np.concatenate([[0], cuts, [n]]).astype(np.int32)
        if k == 1 and int(math.isqrt(n)) ** 2 == n:
            x = gen.grid_points_2d(int(math.isqrt(n)))
        else:
            x = rng.uniform(0, 1, size=(n, 2)).astype(np.float32)
        if siren:
            x = (2.0 * x - 1.0).astype(np.float32)
        return {"params": params, "off": off, "x": x, "q": rng.standard_normal((k, case["r"])) * (0.5 if siren else 1.0)}
    if kind == "recon":
        x = gen.grid_points_2d(case["side"])
        if siren:
            x = (2.0 * x - 1.0).astype(np.float32)
        return {"params": params, "x": x, "q": rng.standard_normal((case["n_codes"], case["r"])) * (0.5 if siren else 1.0)}
    if kind == "fom":
        n, b, model = case["n"], case["batch"], case["model"]
        d = {"ax": None, "ay": None}
        if model == "heat1d":
            d["u"] = np.stack([gen.sine_modes_1d(n, rng)[1] for _ in range(b)])
            d["coef"], d["dt"] = rng.uniform(0.5, 1.0, size=b), 0.25 / (n - 1) ** 2
        elif model.startswith("heat2d"):
            base = np.stack([gen.gaussian_bumps_2d(n, rng) for _ in range(min(b, 4))])
            d["u"] = base[np.arange(b) % len(base)] * rng.uniform(0.5, 1.0, size=(b, 1, 1))
            d["dt"] = 1.0 / (n - 1) ** 2 / 16
            d["coef"] = rng.uniform(0.5, 2.0, size=b)
            if model.endswith("field"):
                strips = gen.piecewise_nu(gen.grid_points_2d(n), [0.0, 0.2, 1.0, 0.2]).reshape(1, n, n)
                d["coef"] = strips * d["coef"].reshape(b, 1, 1)
        else:
            ax, ay = gen.stream_function_faces(n, rng)
            u0 = gen.periodic_bumps_2d(n, rng)
            d["u"] = u0[None] * rng.uniform(0.5, 1.0, size=(b, 1, 1))
            d["ax"], d["ay"] = np.repeat(ax[None], b, axis=0), np.repeat(ay[None], b, axis=0)
            d["coef"], d["dt"] = rng.uniform(1e-3, 1e-2, size=b), 2.5e-4 * min(1.0, (256 / n) ** 1)
        return d
    # train: the encoder's and the decoder's initial parameters, snapshots of bumps, points
    P, r = case["side"] ** 2, case["r"]
    spec = gen.DecoderSpec(case["m"], r, case["width"], case["hidden"])
    lens = [P]
    while (lens[-1] - 6) // 4 + 1 >= 32:
        lens.append((lens[-1] - 6) // 4 + 1)
    parts = [gen.pack_params(gen.xavier_decoder(spec, int(rng.integers(1 << 30))))]
    for _ in lens[1:]:
        parts.append(np.append(rng.standard_normal(6) * math.sqrt(2.0 / 6), 0.0))
    parts += [rng.standard_normal((32, lens[-1])) * math.sqrt(2.0 / (lens[-1] + 32)), np.zeros(32),
              rng.standard_normal((r, 32)) * math.sqrt(2.0 / (32 + r)), np.zeros(r)]
    return {"spec": spec, "lens": lens, "params": np.concatenate([np.asarray(p, np.float32).ravel() for p in parts]),
            "bumps": np.concatenate([rng.uniform(0, 1, (case["B"], 6, 2)), rng.uniform(0.05, 0.12, (case["B"], 6, 1)),
                                     rng.uniform(0.5, 1.0, (case["B"], 6, 1))], axis=2),
            "pts": rng.integers(0, P, size=(case["B"], case["S"])).astype(np.int32)}


def _snapshots(case, d):
    """Standardised bump fields [B][P] and coordinates [P][m] in FP32, formed on the GPU."""
    n = case["side"]
    t = torch.arange(n, device="cuda", dtype=torch.float32) / (n - 1)
    b = _dev(d["bumps"], torch.float32)
    ex = torch.exp(-((t[None, None, :] - b[:, :, 0:1]) ** 2) / (2 * b[:, :, 2:3] ** 2)) * b[:, :, 3:4]
    ey = torch.exp(-((t[None, None, :] - b[:, :, 1:2]) ** 2) / (2 * b[:, :, 2:3] ** 2))
    u = (ex[:, :, :, None] * ey[:, :, None, :]).sum(1).reshape(case["B"], n * n)
    s = float(np.std(np.arange(n) / (n - 1)))
    coords = ((gen.grid_points_2d(n) - 0.5) / s).astype(np.float32)
    return ((u - 0.25) / 0.35).contiguous(), _dev(coords, torch.float32)


def prepare(case, seed):
    d, kind = _inputs(case, seed), case["kind"]
    st = {"case": case}
    if kind in ("step", "decode", "recon"):
        siren = case.get("act") == "siren"
        st["ctx"] = crom.crom_create(case["m"], case["r"], case["width"], case["hidden"],
                                     activation=crom.CROM_ACT_SIREN if siren else crom.CROM_ACT_ELU, omega0=OMEGA0)
        crom.crom_set_weights(st["ctx"], gen.pack_params(d["params"]))
    if kind == "step":
        st["q0"] = _dev(d["q0"], torch.float64)
        st["q"] = torch.empty_like(st["q0"])
        st["status"] = torch.zeros(case["n_inst"], dtype=torch.int32, device="cuda")
        st["args"] = (_dev(d["alpha"], torch.float32), _dev(d["s_off"], torch.int32), _dev(d["samples"], torch.float32))
        st["kw"] = dict(dt=case["dt"], gn_iters=case["gn"], max_samples=int(d["sizes"].max()), precision=PREC[case["prec"]],
                        pde=crom.CROM_PDE_HEAT if case["pde"] == "heat" else crom.CROM_PDE_ADVDIFF,
                        vel=None if d["vel"] is None else _dev(d["vel"], torch.float32),
                        coef_per_sample=case["coef_per_sample"])
    elif kind == "decode":
        rows = _rows(case)
        st["args"] = (_dev(d["q"], torch.float64), _dev(d["off"], torch.int32), _dev(d["x"], torch.float32), case["want"])
        st["out"] = torch.empty((rows, case["n_pts"]), dtype=torch.float32, device="cuda")
    elif kind == "recon":
        st["args"] = (_dev(d["q"], torch.float64), _dev(d["x"], torch.float32))
        st["out"] = torch.empty((case["n_codes"], case["side"] ** 2), dtype=torch.float32, device="cuda")
    elif kind == "fom":
        st["u"] = _dev(d["u"], torch.float32)
        st["tmp"] = torch.empty_like(st["u"])
        st["coef"] = _dev(d["coef"], torch.float32)
        st["kw"] = dict(dt=d["dt"], n_steps=case["steps"], ax=None if d["ax"] is None else _dev(d["ax"], torch.float32),
                        ay=None if d["ay"] is None else _dev(d["ay"], torch.float32))
    else:
        tr = crom.CromTrainer(case["m"], case["r"], case["width"], case["hidden"], case["side"] ** 2, case["B"], case["S"])
        tr.set_precision(PREC[case["prec"]])
        tr.set_params(d["params"])
        st["tr"] = tr
        snaps, coords = _snapshots(case, d)
        st["args"] = (snaps, _dev(d["pts"], torch.int32), coords)
        st["loss"] = torch.zeros(1, dtype=torch.float64, device="cuda")
        st["grads"] = torch.empty(tr.n_params, dtype=torch.float32, device="cuda")
    return st


def _rows(case):
    w, m = case["want"], case["m"]
    return (w & 1) + (m if w & 2 else 0) + (m if w & 4 else 0) + (1 if w & 8 else 0) + (case["r"] if w & 16 else 0)


# ------------------------------------------------------------------ one pass


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "step":
        st["q"].copy_(st["q0"])  # every pass steps from the same codes, as a parameter study does
        if case["steps"]:
            crom.crom_rollout(st["ctx"], st["q"], *st["args"], st["status"], n_steps=case["steps"], **st["kw"])
        else:
            crom.crom_step(st["ctx"], st["q"], *st["args"], st["status"], **st["kw"])
        return {"q": st["q"], "status": st["status"]}
    if kind == "decode":
        if case["prec"] == "fp32":
            crom.crom_decode(st["ctx"], *st["args"], st["out"])
        else:
            crom.crom_decode_tc(st["ctx"], *st["args"], st["out"], precision=PREC[case["prec"]])
        return st["out"]
    if kind == "recon":
        crom.crom_reconstruct(st["ctx"], *st["args"], st["out"], precision=PREC[case["prec"]])
        return st["out"]
    if kind == "fom":
        crom.crom_fom_step(FOM_KIND[case["model"]], st["u"], st["tmp"], st["coef"], **st["kw"])
        return st["u"]
    tr = st["tr"]
    crom.crom_train_step(tr, *st["args"], 1e-4, st["loss"])
    # the gradients on the device, through the C entry point (the binding's get_grads copies to the host)
    crom.raw_call("crom_trainer_get_grads", tr.handle, crom.ctypes.c_void_p(st["grads"].data_ptr()),
                  crom.ctypes.c_size_t(tr.n_params), 1, crom.ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    return {"loss": st["loss"], "grads": st["grads"]}


# ------------------------------------------------------------------ what a pass cannot do without


def _weights(case):
    return gen.param_count(gen.DecoderSpec(case["m"], case["r"], case["width"], case["hidden"]))


def work(case):
    kind = case["kind"]
    if kind == "fom":
        n = case["n"] ** (1 if case["model"] == "heat1d" else 2) * case["batch"]
        per = {"heat1d": 6, "heat2d": 9, "heat2d_field": 10}.get(case["model"], 24)
        arrays = {"heat2d_field": 3}.get(case["model"], 2) + (2 if case["model"].startswith("adv") else 0)
        return {"bytes": 4 * n * arrays, "flops": per * n * case["steps"]}
    m, r, w, L = case["m"], case["r"], case["width"], case["hidden"]
    mat = 2 * (L - 1) * w * w + 2 * w  # one channel through the hidden matrices and the output row
    if kind == "step":
        total = case["n_inst"] * (case["lo"] + case["hi"]) / 2
        # value, dx_1..dx_m and the Laplacian forward and one reverse pass for dg/dq in
        # the first iteration; the value forward and the reverse pass in later ones
        per = (2 + m) * mat + mat + 4 * (m + r) * w + r * (r + 3) + (case["gn"] - 1) * (2 * mat + 4 * (m + r) * w + r * (r + 3))
        b = total * 4 * (m * (2 if case["pde"] == "advdiff" else 1) + (1 if case["coef_per_sample"] else 0))
        b += case["n_inst"] * (16 * r + 12) + 4 * _weights(case)
        return {"bytes": b, "flops": total * per * max(1, case["steps"])}
    if kind == "decode":
        want, n = case["want"], case["n_pts"]
        ch = 1 + (m if want & 14 else 0) + (m if want & 4 else 1 if want & 8 else 0) + (1 if want & 16 else 0)
        return {"bytes": 4 * n * (m + _rows(case)) + 8 * r * case["n_inst"] + 4 * _weights(case),
                "flops": n * (ch * mat + 2 * (m + (r if want & 16 else 0)) * w)}
    if kind == "recon":
        n = case["side"] ** 2
        return {"bytes": 4 * n * (m + case["n_codes"]) + 8 * r * case["n_codes"] + 4 * _weights(case),
                "flops": n * case["n_codes"] * (mat + 2 * m * w)}
    pts = case["B"] * case["S"]
    P = case["side"] ** 2
    return {"bytes": 4 * (case["B"] * P + 2 * P) + 4 * pts + 28 * _weights(case),
            "flops": pts * 3 * (mat + 2 * m * w) + 2 * case["B"] * P * 9}


# ------------------------------------------------------------------ the same in 64 bits


def _act(z, siren):
    """s(z), s'(z), s''(z)."""
    if siren:
        sn, cs = torch.sin(OMEGA0 * z), torch.cos(OMEGA0 * z)
        return sn, OMEGA0 * cs, -OMEGA0 ** 2 * sn
    e = torch.exp(z.clamp(max=0.0))
    pos = z > 0
    return torch.where(pos, z, torch.expm1(z.clamp(max=0.0))), torch.where(pos, 1.0, e), torch.where(pos, 0.0, e)


def _network(params, siren, x, q, first, second, jac):
    """Value, dg/dx_k (first), d2g/dx_k^2 (second) and dg/dq (jac) at points x [N][m] with codes q [N][r]."""
    m = x.shape[1]
    W = [w for w, _ in params]
    z = torch.cat([x, q], 1) @ W[0].T + params[0][1]
    dz = [W[0][:, k].expand_as(z) for k in range(m)] if first or second else []
    d2z = [torch.zeros_like(z) for _ in range(m)] if second else []
    slopes = []
    for layer in range(1, len(W)):
        h, s1, s2 = _act(z, siren)
        if jac:
            slopes.append(s1)
        d2h = [s2 * dz[k] ** 2 + s1 * d2z[k] for k in range(m)] if second else []
        dh = [s1 * a for a in dz]
        z = h @ W[layer].T + params[layer][1]
        dz, d2z = [a @ W[layer].T for a in dh], [a @ W[layer].T for a in d2h]
    out = {"val": z[:, 0], "dx": [a[:, 0] for a in dz], "dxx": [a[:, 0] for a in d2z]}
    if jac:
        delta = W[-1].expand(x.shape[0], -1) * slopes[-1]
        for layer in range(len(W) - 2, 0, -1):
            delta = (delta @ W[layer]) * slopes[layer - 1]
        out["dq"] = delta @ W[0][:, m:]
    return out


def _f64(params):
    return [(_dev(w, torch.float64), _dev(b, torch.float64)) for w, b in params]


def _exact_step(case, d):
    siren, m, n = case["act"] == "siren", case["m"], case["n_inst"]
    params = _f64(d["params"])
    x = _dev(d["samples"], torch.float64)
    inst = _dev(np.repeat(np.arange(n), d["sizes"]), torch.int64)
    alpha = _dev(d["alpha"], torch.float64)
    alpha = alpha if case["coef_per_sample"] else alpha[inst]
    vel = None if d["vel"] is None else _dev(d["vel"], torch.float64)
    q = _dev(d["q0"], torch.float64)
    r, N, chunk = case["r"], x.shape[0], 1 << 15

    def over(fn):
        parts = [fn(slice(a, min(N, a + chunk))) for a in range(0, N, chunk)]
        return [torch.cat(p) for p in zip(*parts)]

    for _ in range(max(1, case["steps"])):
        qn = q

        def start(s):
            o = _network(params, siren, x[s], qn[inst[s]], True, True, True)
            f = alpha[s] * sum(o["dxx"])
            if vel is not None:
                f = f - sum(vel[s, k] * o["dx"][k] for k in range(m))
            return o["val"], case["dt"] * f, o["dq"]

        base, df, J = over(start)
        res = -df
        for it in range(case["gn"]):
            if it:
                def later(s):
                    o = _network(params, siren, x[s], q[inst[s]], False, False, True)
                    return o["val"], o["dq"]
                val, J = over(later)
                res = (val - base) - df
            A = torch.zeros(n, r, r, dtype=torch.float64, device="cuda")
            g = torch.zeros(n, r, dtype=torch.float64, device="cuda")
            for a in range(0, N, chunk):
                s = slice(a, min(N, a + chunk))
                A.index_add_(0, inst[s], J[s, :, None] * J[s, None, :])
                g.index_add_(0, inst[s], J[s] * res[s, None])
            q = q - torch.linalg.solve(A, g)
    return {"q": q, "status": None}


def _exact_fom(case, d):
    u = _dev(d["u"], torch.float32).double()
    coef = _dev(d["coef"], torch.float32).double()
    n, dt, model = case["n"], d["dt"], case["model"]
    if model == "heat1d":
        for _ in range(case["steps"]):
            v = torch.zeros_like(u)
            v[:, 1:-1] = u[:, 1:-1] + dt * (n - 1) ** 2 * coef[:, None] * (u[:, :-2] + u[:, 2:] - 2 * u[:, 1:-1])
            u = v
        return u
    if model.startswith("heat2d"):
        coef = coef if model.endswith("field") else coef[:, None, None]
        for _ in range(case["steps"]):
            p = torch.nn.functional.pad(u[:, None], (1, 1, 1, 1), mode="reflect")[:, 0]
            lap = p[:, :-2, 1:-1] + p[:, 2:, 1:-1] + p[:, 1:-1, :-2] + p[:, 1:-1, 2:] - 4 * u
            u = u + dt * (n - 1) ** 2 * coef * lap
        return u
    ax, ay = _dev(d["ax"], torch.float32).double(), _dev(d["ay"], torch.float32).double()

    def flux(a, left, right):
        return a * 0.5 * (left + right) if model.endswith("central") else a * torch.where(a > 0, left, right)

    for _ in range(case["steps"]):
        fx = flux(ax, u, u.roll(-1, 1))
        fy = flux(ay, u, u.roll(-1, 2))
        div = (fx - fx.roll(1, 1) + fy - fy.roll(1, 2)) * n
        lap = (u.roll(1, 1) + u.roll(-1, 1) + u.roll(1, 2) + u.roll(-1, 2) - 4 * u) * n * n
        u = u + dt * (coef[:, None, None] * lap - div)
    return u


def _exact_train(case, d):
    snaps, coords = (t.double() for t in _snapshots(case, d))
    p = _dev(d["params"], torch.float64).requires_grad_()
    at = 0

    def take(*shape):
        nonlocal at
        size = int(np.prod(shape))
        at += size
        return p[at - size:at].view(*shape)

    dims = d["spec"].dims
    dec = [(take(dims[k + 1], dims[k]), take(dims[k + 1])) for k in range(len(dims) - 1)]
    h = snaps
    for _ in d["lens"][1:]:
        w, b = take(6), take(1)
        h = torch.nn.functional.elu(h.unfold(1, 6, 4) @ w + b)
    w, b = take(32, d["lens"][-1]), take(32)
    h = torch.nn.functional.elu(h @ w.T + b)
    w, b = take(case["r"], 32), take(case["r"])
    q = h @ w.T + b
    pts = _dev(d["pts"], torch.int64)
    target = torch.gather(snaps, 1, pts)
    m, total = case["m"], pts.numel()
    loss = torch.zeros((), dtype=torch.float64, device="cuda")
    h = coords[pts] @ dec[0][0][:, :m].T + (q @ dec[0][0][:, m:].T + dec[0][1])[:, None, :]
    for k in range(1, len(dec)):
        h = torch.nn.functional.elu(h) @ dec[k][0].T + dec[k][1]
    loss = ((h[..., 0] - target) ** 2).sum() / total
    loss.backward()
    return {"loss": loss.detach().reshape(1), "grads": p.grad}


def exact(case, seed):
    d, kind = _inputs(case, seed), case["kind"]
    if kind == "step":
        return _exact_step(case, d)
    if kind == "fom":
        return _exact_fom(case, d)
    if kind == "train":
        return _exact_train(case, d)
    params, siren = _f64(d["params"]), case["act"] == "siren"
    x, q, chunk = _dev(d["x"], torch.float64), _dev(d["q"], torch.float64), 1 << 16
    if kind == "decode":
        want, rows = case["want"], []
        inst = _dev(np.repeat(np.arange(case["n_inst"]), np.diff(d["off"])), torch.int64)
        for a in range(0, x.shape[0], chunk):
            s = slice(a, a + chunk)
            o = _network(params, siren, x[s], q[inst[s]], bool(want & 2), bool(want & 12), bool(want & 16))
            c = [o["val"]] if want & 1 else []
            c += o["dx"] if want & 2 else []
            c += o["dxx"] if want & 4 else []
            c += [sum(o["dxx"])] if want & 8 else []
            c += list(o["dq"].T) if want & 16 else []
            rows.append(torch.stack(c))
        return torch.cat(rows, 1)
    out = torch.empty(case["n_codes"], x.shape[0], dtype=torch.float64, device="cuda")
    for k in range(case["n_codes"]):
        for a in range(0, x.shape[0], chunk):
            xs = x[a:a + chunk]
            out[k, a:a + chunk] = _network(params, siren, xs, q[k].expand(xs.shape[0], -1), False, False, False)["val"]
    return out
