"""The work whose speed is measured: calls that a user of the library makes, over the range of their sizes.

A case is a dict of plain values.  `listed()` names the standing ones, `draw(rng)` gives another of the
same ranges, `prepare(case, seed)` makes what a program holds before the call (fields on the device or in
page-locked host memory, output buffers, a `Labeller`), and `run(state)` is one pass through the public
entry points.  Fields are synthetic, with the structure of the paper's: random sites (percolation, the
hardest partition), emulsion droplets and bijels (Sec. 5), capsule index fields (Sec. 6) and the block
pattern of the paper's own benchmark (Sec. 3).  Every output is a whole number, so there is nothing to
compare in 64 bits.
"""
import math

import numpy as np
import torch

from paper_1405_1931_gb300 import fields, hk

P_C = fields.P_C_SIMPLE_CUBIC


def listed():
    return [
        # One call on the smallest lattice that is used in earnest: latency.
        {"name": "small_32", "kind": "iid", "nx": 32, "ny": 32, "nz": 32, "p": 0.3, "px": 1, "py": 1, "pz": 1},
        # An emulsion snapshot of an ordinary simulation, 600 droplets.
        {"name": "emulsion_256", "kind": "emulsion", "nx": 256, "ny": 256, "nz": 256, "droplets": 600,
         "px": 1, "py": 1, "pz": 1},
        # A box whose sides divide into nothing (rows not 16-byte aligned), periodic along two axes.
        {"name": "ragged_iid", "kind": "iid", "nx": 387, "ny": 283, "nz": 221, "p": P_C, "px": 1, "py": 0, "pz": 1},
        # A bijel: two labyrinthine phases, one cluster through everything.
        {"name": "bijel_512", "kind": "waves", "nx": 512, "ny": 512, "nz": 512, "wavelength": 24.0,
         "px": 1, "py": 1, "pz": 1},
        # The paper's benchmark: alternating blocks that touch only at their edges.
        {"name": "blocks_1024", "kind": "blocks", "nx": 1024, "ny": 1024, "nz": 1024, "b": 16,
         "px": 1, "py": 1, "pz": 1},
        # The headline: a large lattice at the percolation threshold, 56 million clusters.
        {"name": "critical_1024", "kind": "iid", "nx": 1024, "ny": 1024, "nz": 1024, "p": P_C,
         "px": 1, "py": 1, "pz": 1},
        # Many uneven lattices in one call (a parameter study).
        {"name": "batch_96", "kind": "batch", "n": 96, "shapes": 2, "lo": 32, "hi": 384, "step": 16},
        # What the server packs into one call: emulsion requests of up to 128 sites a side.
        {"name": "batch_served", "kind": "served", "n": 14, "shapes": 3, "lo": 64, "hi": 128},
        # The interior of every capsule of a large suspension, computed anew.
        {"name": "interior_state_1024", "kind": "state", "nx": 1024, "ny": 1024, "nz": 1024, "cell": 113,
         "px": 1, "py": 1, "pz": 1},
        # Labels, sizes and interior/exterior tags of a smaller suspension.
        {"name": "label_interior_256", "kind": "interior", "nx": 256, "ny": 256, "nz": 256, "cell": 85,
         "px": 1, "py": 1, "pz": 1},
        # The step of every time step between two refreshes: membranes have moved a little.
        {"name": "interior_update_1024", "kind": "update", "nx": 1024, "ny": 1024, "nz": 1024, "cell": 113,
         "px": 1, "py": 1, "pz": 1},
        # A field in host memory, labelled and brought back.
        {"name": "host_256", "kind": "host", "nx": 256, "ny": 256, "nz": 256, "p": P_C, "px": 1, "py": 1, "pz": 1},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _box(rng, lo, hi):
    """Sides around one log-uniform scale in [lo, hi], each off by up to a factor 1.6; a third of the boxes
    have rows of a multiple of four sites, the others any length."""
    side = _log(rng, lo, hi)
    d = [max(lo, min(hi, int(round(side * _log(rng, 1 / 1.6, 1.6))))) for _ in range(3)]
    if rng.random() < 1 / 3:
        d[0] = max(4, d[0] // 4 * 4)
    return {"nx": d[0], "ny": d[1], "nz": d[2], "px": rng.randint(0, 1), "py": rng.randint(0, 1),
            "pz": rng.randint(0, 1)}


def draw(rng):
    kind = rng.choice(["iid", "iid", "iid", "emulsion", "waves", "blocks", "batch", "served", "state", "interior",
                       "update", "host"])
    if kind == "iid":
        return {"kind": kind, "p": round(rng.uniform(0.15, 0.45), 3), **_box(rng, 16, 960)}
    if kind == "emulsion":
        b = _box(rng, 64, 512)
        sites = b["nx"] * b["ny"] * b["nz"]
        return {"kind": kind, "droplets": max(1, int(sites * rng.uniform(0.1, 0.3) / 5236.0)), **b}
    if kind == "waves":
        return {"kind": kind, "wavelength": round(rng.uniform(12.0, 40.0), 1), **_box(rng, 64, 640)}
    if kind == "blocks":
        return {"kind": kind, "b": rng.choice([2, 4, 8, 16, 32, 64, 128]), **_box(rng, 128, 1024)}
    if kind == "batch":
        lo = rng.choice([16, 32, 48])
        return {"kind": kind, "n": int(round(_log(rng, 8, 96))), "shapes": rng.randrange(1000), "lo": lo,
                "hi": rng.choice([64, 128, 256, 384]), "step": rng.choice([1, 16])}
    if kind == "served":
        return {"kind": kind, "n": rng.randint(2, 24), "shapes": rng.randrange(1000), "lo": 64, "hi": 128}
    if kind == "host":
        return {"kind": kind, "p": round(rng.uniform(0.15, 0.45), 3), **_box(rng, 32, 320)}
    return {"kind": kind, "cell": rng.randint(48, 128), **_box(rng, 96, 960)}


# ---- fields -------------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _iid(nx, ny, nz, p, seed):
    phi = torch.rand((nz, ny, nx), generator=_gen(seed), device="cuda")
    return phi.sub_(1.0 - p)


def _emulsion(nx, ny, nz, droplets, seed):
    phi = torch.empty((nz, ny, nx), dtype=torch.float32, device="cuda")
    centres, radii = fields.sphere_params(droplets, (nx, ny, nz), seed)
    rc = hk.hk_gen_spheres(phi.data_ptr(), nx, ny, nz, centres, radii, 8.0, torch.cuda.current_stream().cuda_stream)
    assert rc == 0
    return phi


def _waves(nx, ny, nz, wavelength, seed, waves=24):
    """A sum of plane waves of one length in random directions, periodic in the box: its sign divides the box
    into two labyrinths.  Each wave factors over z and (y, x), so the sum is one matrix product."""
    r = np.random.default_rng(seed)
    v = r.normal(size=(waves, 3))
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    dims = np.array([nx, ny, nz], dtype=np.float64)
    k = 2.0 * np.pi * np.round(v * dims / wavelength) / dims
    phase = r.uniform(0.0, 2.0 * np.pi, size=waves)
    ax = [torch.arange(n, dtype=torch.float64, device="cuda") for n in (nx, ny, nz)]
    kx, ky, kz = (torch.from_numpy(np.ascontiguousarray(k[:, a])).cuda()[:, None] for a in range(3))
    yx = ((ky * ax[1])[:, :, None] + (kx * ax[0])[:, None, :] + torch.from_numpy(phase).cuda()[:, None, None])
    yx = yx.reshape(waves, ny * nx)
    z = kz * ax[2]
    left = torch.cat([torch.cos(z), -torch.sin(z)]).float().t().contiguous()
    right = torch.cat([torch.cos(yx), torch.sin(yx)]).float()
    return (left @ right).reshape(nz, ny, nx)


def _blocks(nx, ny, nz, b, seed):
    off = np.random.default_rng(seed).integers(0, 2 * b, 3).tolist()
    par = [(((torch.arange(n, device="cuda") + o) % n) // b % 2).to(torch.int8) for n, o in zip((nx, ny, nz), off)]
    s = (par[2].view(nz, 1, 1) + par[1].view(1, ny, 1) + par[0].view(1, 1, nx)) & 1
    return 1.0 - 2.0 * s.to(torch.float32)


def _capsules(nx, ny, nz, cell, seed):
    """One ellipsoid in each cell of a coarse grid: per cell and axis its centre and semi-axis."""
    g = [max(1, n // cell) for n in (nz, ny, nx)]
    room = min(n // k for n, k in zip((nz, ny, nx), g))
    hi = max(4.0, min(30.0, room / 2 - 4.0))
    lo = min(8.0, hi / 2)
    r = np.random.default_rng(seed)
    axes = lo + (hi - lo) * r.random((3, *g))
    centres = np.empty((3, *g))
    for a, (n, k) in enumerate(zip((nz, ny, nx), g)):
        w = n / k
        first = (np.arange(k) * w).reshape([k if i == a else 1 for i in range(3)])
        free = np.maximum(w - 2 * (axes[a] + 3.0), 0.0)
        centres[a] = first + (w - free) / 2 + free * r.random(g)
    return centres, axes


def _inside(nx, ny, nz, capsules):
    """True on the sites of the ellipsoids."""
    centres, axes = (torch.from_numpy(v).float().cuda() for v in capsules)
    g = centres.shape[1:]
    of = [torch.div(torch.arange(n, device="cuda") * k, n, rounding_mode="floor") for n, k in zip((nz, ny, nx), g)]
    at = [torch.arange(n, dtype=torch.float32, device="cuda") for n in (nz, ny, nx)]
    out = torch.empty((nz, ny, nx), dtype=torch.bool, device="cuda")
    for i in range(g[0]):
        z = [j for j in range(-(-i * nz // g[0]), -(-(i + 1) * nz // g[0]))]
        c = [centres[a, i][of[1]][:, of[2]] for a in range(3)]
        s = [1.0 / axes[a, i][of[1]][:, of[2]] for a in range(3)]
        plane = ((at[1][:, None] - c[1]) * s[1]) ** 2 + ((at[2][None, :] - c[2]) * s[2]) ** 2
        out[z[0]:z[-1] + 1] = ((at[0][z[0]:z[-1] + 1, None, None] - c[0]) * s[0]) ** 2 + plane <= 1.0
    return out


def _index(inside):
    """The index field of Sec. 6: -0.25 on the inner and 0.25 on the outer layer of every membrane, else -1."""
    grown, core = inside.clone(), inside.clone()
    for a in range(3):
        n = inside.shape[a]
        for d, s in ((slice(1, n), slice(0, n - 1)), (slice(0, n - 1), slice(1, n))):
            dst, src = [slice(None)] * 3, [slice(None)] * 3
            dst[a], src[a] = d, s
            grown[tuple(dst)] |= inside[tuple(src)]
            core[tuple(dst)] &= inside[tuple(src)]
    index = torch.full(inside.shape, -1.0, device="cuda")
    index.masked_fill_(grown & ~inside, 0.25)
    return index.masked_fill_(inside & ~core, -0.25)


# ---- state --------------------------------------------------------------------------------------

_labeller = None


def _lab():
    """The context a program opens once and keeps."""
    global _labeller
    if _labeller is None:
        _labeller = hk.Labeller(0)
    return _labeller


def _outputs(sites, n=1):
    """Output buffers of n lattices back to back: labels, sizes, histograms and counts (sizes beyond the count
    are not written, so they start as zeros)."""
    return (torch.empty(sites, dtype=torch.int32, device="cuda"),
            torch.zeros(max(1, (sites + n) // 2), dtype=torch.int64, device="cuda"),
            torch.empty((n, 32), dtype=torch.int64, device="cuda"), torch.empty(n, dtype=torch.int64, device="cuda"))


def _sides(case):
    """The shapes, occupancies and periodic edges of a batch, from its `shapes` number."""
    r = np.random.default_rng(case["shapes"])
    lo, hi, out = case["lo"], case["hi"], []
    for _ in range(case["n"]):
        if case["kind"] == "served":   # cubes, log-uniform, periodic
            side = int(round(lo * (hi / lo) ** r.random()))
            out.append(((side,) * 3, 0.3, (1, 1, 1)))
        else:
            step = case["step"]
            dims = tuple(int(lo + step * r.integers(0, (hi - lo) // step + 1)) for _ in range(3))
            out.append((dims, 0.15 + 0.3 * r.random(), tuple(int(v) for v in r.integers(0, 2, 3))))
    return out


def _prepare_batch(case, seed):
    shapes = _sides(case)
    pad = [-(-int(np.prod(d)) // 128) * 128 for d, _, _ in shapes]   # every lattice starts aligned
    labels, sizes, hist, ncl = _outputs(sum(pad), len(shapes))
    labels.zero_()
    items, at = [], 0
    for i, ((dims, p, per), room) in enumerate(zip(shapes, pad)):
        nx, ny, nz = dims
        n, cap = nx * ny * nz, (nx * ny * nz + 1) // 2
        if case["kind"] == "served":   # droplets of 5236 sites on average, a volume fraction of 0.3
            phi = _emulsion(nx, ny, nz, max(1, int(round(p * n / 5236.0))), seed * 128 + i)
        else:
            phi = _iid(nx, ny, nz, p, seed * 128 + i)
        items.append((phi, per, (labels[at:at + n].view(nz, ny, nx), sizes[at // 2:at // 2 + cap], hist[i],
                                 ncl[i:i + 1], cap)))
        at += room
    return {"lab": _lab(), "items": items, "out": (labels, sizes, hist, ncl)}


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("batch", "served"):
        return {"kind": "batch", **_prepare_batch(case, seed)}
    dims = (case["nx"], case["ny"], case["nz"])
    nx, ny, nz = dims
    s = {"kind": kind, "lab": _lab(), "per": (case["px"], case["py"], case["pz"])}
    if kind in ("state", "interior", "update"):
        centres, axes = _capsules(nx, ny, nz, case["cell"], seed)
        inside = _inside(nx, ny, nz, (centres, axes))
        if kind == "update":   # the state of the step before, then every membrane moves by up to a quarter site
            s["state"] = inside.to(torch.int8)
            move = np.random.default_rng(seed + 1).uniform(-0.25, 0.25, centres.shape)
            inside = _inside(nx, ny, nz, (centres + move, axes))
        else:
            s["state"] = torch.empty((nz, ny, nx), dtype=torch.int8, device="cuda")
        s["field"] = _index(inside)
    elif kind == "emulsion":
        s["field"] = _emulsion(nx, ny, nz, case["droplets"], seed)
    elif kind == "waves":
        s["field"] = _waves(nx, ny, nz, case["wavelength"], seed)
    elif kind == "blocks":
        s["field"] = _blocks(nx, ny, nz, case["b"], seed)
    else:
        s["field"] = _iid(nx, ny, nz, case["p"], seed)
    if kind == "host":
        n = nx * ny * nz
        s["field"] = s["field"].cpu().pin_memory()
        s["out"] = (torch.empty((nz, ny, nx), dtype=torch.int32).pin_memory(),
                    torch.zeros((n + 1) // 2, dtype=torch.int64).pin_memory(),
                    torch.empty(32, dtype=torch.int64).pin_memory(), torch.empty(1, dtype=torch.int64).pin_memory())
    elif kind not in ("state", "update"):
        labels, sizes, hist, ncl = _outputs(nx * ny * nz)
        s["out"] = (labels.view(nz, ny, nx), sizes, hist[0], ncl, (nx * ny * nz + 1) // 2)
        if kind == "interior":   # a program knows how many capsules it holds
            s["clusters"] = int(_lab().label(-0.5 - s["field"], s["per"])[3].item())
    return s


def run(state):
    kind, lab = state["kind"], state["lab"]
    if kind == "batch":
        lab.label_batched(state["items"])
        return state["out"]
    if kind == "state":
        return lab.interior_state(state["field"], state["per"], out=state["state"])
    if kind == "update":
        return hk.interior_update(state["state"], state["field"])
    if kind == "interior":
        labels, sizes, hist, ncl, inside = lab.label_interior(state["field"], state["per"], out=state["out"])
        return labels, sizes, hist, ncl, inside[:state["clusters"]]   # tags beyond the count are not written
    if kind == "host":
        labels, sizes, hist, ncl = state["out"]
        lab.label_host_async(state["field"], labels, sizes, hist, ncl, state["per"])
        return labels, sizes, hist, ncl
    return lab.label(state["field"], state["per"], out=state["out"])


def _clusters(n, p):
    """About how many clusters n random sites of occupancy p have: sites - bonds + plaquettes, and never fewer
    than the single sites."""
    return n * max(p - 3 * p ** 2 + 3 * p ** 4, p * (1 - p) ** 6)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        dims = [(int(np.prod(d)), p) for d, p, _ in _sides(case)]
        return {"bytes": sum(8 * n + 8 * _clusters(n, p) + 264 for n, p in dims), "flops": 0}
    if kind == "served":
        return {"bytes": sum(8 * int(np.prod(d)) + 264 for d, _, _ in _sides(case)), "flops": 0}
    n = case["nx"] * case["ny"] * case["nz"]
    if kind == "state":      # the index field read, a byte a site written
        return {"bytes": 5 * n, "flops": 0}
    if kind == "update":     # the index field and the old state read, the new state written
        return {"bytes": 6 * n, "flops": 0}
    clusters = {"iid": lambda: _clusters(n, case["p"]), "host": lambda: _clusters(n, case["p"]),
                "blocks": lambda: n / (2 * case["b"] ** 3)}.get(kind, lambda: 0)()
    return {"bytes": 8 * n + 8 * clusters + 264, "flops": 0}   # field read, labels, sizes, histogram and count written
