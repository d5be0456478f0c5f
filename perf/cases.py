"""Timed cases of the imaging library: the work its users have it do, through
the binding's public calls, over the range of sizes the paper's arrays span.

A case is one cadence of one path.  Station sizes follow the uneven array's
rule (diameter 38 m sqrt(N_e / 256), 1.5 m minimum spacing, lambda 3 m, cells
of half a wavelength, 3 x 3 Gaussian taps, grid side from the padding factor
2), so 64, 256 and 700 elements give the 32^2, 64^2 and 128^2 grids; the dense
all-sky lattice has one unit tap per element.  A program keeps its context,
layouts and plan from cadence to cadence, so prepare() makes them.
"""
from __future__ import annotations

import functools
import math
import weakref

import numpy as np
import torch

from paper_2411_17804_gb300 import hai
from paper_2411_17804_gb300 import inputs as I

PREC = {"fp32": hai.HAI_PREC_FP32, "fp16": hai.HAI_PREC_FP16, "fp16_split": hai.HAI_PREC_FP16_SPLIT,
        "bf16": hai.HAI_PREC_BF16, "bf16_split": hai.HAI_PREC_BF16_SPLIT}
UNEVEN = I.UnevenConfig()
HIER = I.HierarchyConfig()


def listed():
    return [
        # the smallest call: one channel, one polarisation of a 64-element
        # station at full precision, where launches and latency count
        {"name": "station64_fp32", "kind": "epic", "array": "disk", "elements": 64, "pols": 1, "channels": 1,
         "samples": 1024, "prec": "fp32"},
        # one cadence of an SKA-low station on tensor cores, the usual call
        {"name": "ska_fp16", "kind": "epic", "array": "disk", "elements": 256, "pols": 2, "channels": 64,
         "samples": 2048, "prec": "fp16"},
        # a ragged part of it at full precision: a station with elements out of
        # service, a sub-band, a cadence that no tile divides
        {"name": "ska_ragged_fp32", "kind": "epic", "array": "disk", "elements": 251, "pols": 2, "channels": 37,
         "samples": 999, "prec": "fp32"},
        # the dense all-sky lattice on tensor cores: the headline's work, the largest
        {"name": "dense_fp16", "kind": "epic", "array": "lattice", "side": 128, "pols": 2, "channels": 16,
         "samples": 1000, "prec": "fp16"},
        # the same at full precision, a short cadence
        {"name": "dense_fp32", "kind": "epic", "array": "lattice", "side": 128, "pols": 2, "channels": 16,
         "samples": 100, "prec": "fp32"},
        # coherent imaging between stations: one beam of the core on 128^2
        {"name": "core_epic_fp16", "kind": "epic", "array": "stations", "elements": 256, "pols": 2, "channels": 32,
         "samples": 1000, "prec": "fp16"},
        # correlator and FFT imager of the SKA-low station, the alternative to EPIC
        {"name": "ska_corr_xfft", "kind": "corr_xfft", "elements": 256, "pols": 2, "channels": 64, "samples": 2048},
        # station beams of the hierarchical array (a quarter of its stations),
        # 16 beams requantised to int8
        {"name": "beamform_int8", "kind": "beamform", "stations": 64, "elements": 256, "pols": 2, "channels": 32,
         "samples": 1000, "beams": 16, "shift": 11},
        # its inter-station stage: beams reordered, correlated, imaged on 256^2
        {"name": "core_xfft", "kind": "interstation", "stations": 256, "beams": 16, "channels": 32, "samples": 1000,
         "grid": 256},
        # the pairs that grid drops, imaged by the direct sum
        {"name": "tail_xbf", "kind": "xbf", "stations": 256, "beams": 4, "channels": 32, "grid": 256, "prec": "fp16"},
        # gridded visibilities back from the lattice's accumulated images
        {"name": "fft_correlator", "kind": "fftcorr", "grid": 512, "pols": 2, "channels": 16},
        # an array of uneven stations, both levels of the hierarchy in one launch
        {"name": "uneven_plan", "kind": "plan", "stations": 96, "channels": 32, "samples": 64, "beams": 4},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["epic", "epic", "epic", "lattice", "stations", "corr_xfft", "beamform", "interstation", "xbf",
                       "fftcorr", "plan"])
    if kind == "epic":        # stations of 16 to 1024 elements, every precision
        n = _log(rng, 16, 1024)
        prec = rng.choice(["fp32", "fp32", "fp16", "fp16", "fp16_split", "bf16", "bf16_split"])
        if prec == "fp32" and I.uneven_grid_side(n, UNEVEN) == 128:
            t = _log(rng, 32, 256)
        else:
            t = _log(rng, 64, 2048)
        return {"kind": "epic", "array": "disk", "elements": n, "pols": rng.choice([1, 2]) if prec == "fp32" else 2,
                "channels": _log(rng, 1, 64), "samples": t, "prec": prec}
    if kind == "lattice":     # 256^2 and 512^2 grids
        prec = rng.choice(["fp32", "fp16", "fp16", "fp16_split", "bf16"])
        return {"kind": "epic", "array": "lattice", "side": rng.randint(40, 128), "pols": 2, "channels": _log(rng, 1, 16),
                "samples": _log(rng, 16, 400 if prec in ("fp16", "bf16") else 128), "prec": prec}
    if kind == "stations":
        return {"kind": "epic", "array": "stations", "elements": _log(rng, 64, 512), "pols": 2,
                "channels": _log(rng, 2, 48), "samples": _log(rng, 100, 1000), "prec": rng.choice(["fp16", "fp16", "bf16"])}
    if kind == "corr_xfft":
        return {"kind": "corr_xfft", "elements": _log(rng, 16, 300), "pols": rng.choice([1, 2, 2]),
                "channels": _log(rng, 2, 64), "samples": _log(rng, 64, 2048)}
    if kind == "beamform":
        return {"kind": "beamform", "stations": _log(rng, 2, 64), "elements": 8 * _log(rng, 4, 40), "pols": 2,
                "channels": _log(rng, 2, 32), "samples": _log(rng, 64, 1000), "beams": rng.choice([8, 16, 16]),
                "shift": rng.choice([-1, 11])}
    if kind == "interstation":
        return {"kind": "interstation", "stations": _log(rng, 32, 320), "beams": rng.choice([1, 4, 9, 16]),
                "channels": _log(rng, 2, 32), "samples": _log(rng, 100, 1000), "grid": rng.choice([128, 256])}
    if kind == "xbf":
        return {"kind": "xbf", "stations": _log(rng, 64, 280), "beams": rng.choice([1, 4]), "channels": _log(rng, 2, 32),
                "grid": rng.choice([128, 256]), "prec": rng.choice(["fp16", "fp16_split"])}
    if kind == "fftcorr":
        return {"kind": "fftcorr", "grid": rng.choice([32, 64, 128, 256, 512]), "pols": rng.choice([1, 2, 2]),
                "channels": _log(rng, 2, 64) if rng.random() < 0.7 else 16}
    return {"kind": "plan", "stations": _log(rng, 12, 96), "channels": _log(rng, 4, 32), "samples": _log(rng, 32, 64),
            "beams": rng.choice([1, 4])}


# ------------------------------------------------------------------ geometry
@functools.lru_cache(maxsize=None)
def _station(n_elem: int):
    """(element positions, anchors, taps, grid side) of a station by the uneven array's rule."""
    cfg = I.uneven_station(UNEVEN, n_elem, n_elem)
    pos = I.station_layout(cfg)
    anchors, taps = I.station_kernel(cfg, pos)
    return pos, anchors, taps, cfg.grid_n


@functools.lru_cache(maxsize=4)
def _lattice(side: int):
    lam = I.DENSE_ALLSKY_16384.lam_m
    pos = I.lattice_layout(side, 0.5 * lam)
    n = 512 if side > 64 else 256
    anchors, taps = I.unit_kernel(pos, lam, 0.5, n)
    return pos, anchors, taps, n


@functools.lru_cache(maxsize=8)
def _centres(n_station: int):
    """Station centres of the hierarchical array: a 1 km core and a tail of one station in eight."""
    cfg = I.HierarchyConfig(n_station=n_station, n_tail=max(1, n_station // 8),
                            core_diameter_m=1000.0 * max(1.0, math.sqrt(n_station / 256.0)))
    return I.station_centres(cfg)


@functools.lru_cache(maxsize=8)
def _uneven(n_station: int):
    """(element counts, centres) of the uneven array's first stations."""
    return [int(n) for n in I.uneven_station_sizes(UNEVEN)[:n_station]], I.uneven_centres(UNEVEN, n_station)


def _beam_dirs(n_beam: int):
    return I.beam_directions(n_beam, HIER.station.lam_m, HIER.station.diameter_m)


# ------------------------------------------------------------------ inputs
def _sky(seed: int, n_src: int = 20, reach: float = 0.8):
    return I.draw_sources(n_src, np.random.default_rng(seed), max_dircos=reach)


def _noise(shape, seed: int):
    """Quantised noise voltages of rms 18 counts, in slices of the first axis."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    out = torch.empty(shape, dtype=torch.int8, device="cuda")
    for s in range(shape[0]):
        x = torch.randn(shape[1:], generator=gen, device="cuda", dtype=torch.float16)
        out[s] = (x * 18.0).round_().clamp_(-127, 127).to(torch.int8)
    return out


def _beams(case, seed: int, extent: float):
    """Station beams towards each direction, [K][C][T][P][S][2]: a few sources
    inside the station beam above the noise, as the beamformer returns them."""
    pos = _centres(case["stations"] if "stations" in case else case["elements"])
    dirs, flux = _sky(seed, 5, extent)
    k = case.get("beams", 1)
    v = I.voltages(pos, HIER.station.lam_m, dirs, flux, k * case["channels"], case["samples"], 2, seed, device="cuda")
    return v.view(k, case["channels"], case["samples"], 2, len(pos), 2)


# ------------------------------------------------------------------ handles
@functools.lru_cache(maxsize=1)
def _ctx():
    return hai.hai_create(torch.cuda.current_device())


class _State(dict):
    """Inputs, outputs and handles of one program; the handles go with it."""

    def own(self, handle, destroy):
        weakref.finalize(self, destroy, handle)
        return handle


def prepare(case, seed):
    s = _State(case=case)
    return _PREPARE[case["kind"]](case, seed, s)


def run(state):
    return _RUN[state["case"]["kind"]](state)


def _prepare_epic(case, seed, s):
    C, T, P = case["channels"], case["samples"], case["pols"]
    if case["array"] == "stations":
        pos, n = _centres(case["elements"]), 128
        lay, _ = hai.hai_station_epic_layout_create(_ctx(), pos, HIER.station.lam_m, HIER.cell_m, n, _beam_dirs(16), 5, P)
        s["volt"] = _beams(case, seed, 0.03)[0]
    else:
        pos, anchors, taps, n = _station(case["elements"]) if case["array"] == "disk" else _lattice(case["side"])
        lay = hai.hai_layout_create(_ctx(), anchors, taps, n, P)
        lam = UNEVEN.lam_m if case["array"] == "disk" else I.DENSE_ALLSKY_16384.lam_m
        s["volt"] = I.voltages(pos, lam, *_sky(seed), C, T, P, seed, device="cuda")
    s["layout"] = s.own(lay, hai.hai_layout_destroy)
    s["img"] = torch.empty((C, 4 if P == 2 else 1, n, n), device="cuda")
    return s


def _run_epic(s):
    c = s["case"]
    hai.hai_epic_image(_ctx(), s["layout"], s["volt"], c["channels"], c["samples"], PREC[c["prec"]], s["img"])
    return s["img"]


def _prepare_corr_xfft(case, seed, s):
    C, T, P, ne = case["channels"], case["samples"], case["pols"], case["elements"]
    pos, anchors, taps, n = _station(ne)
    s["layout"] = s.own(hai.hai_layout_create(_ctx(), anchors, taps, n, P), hai.hai_layout_destroy)
    s["volt"] = I.voltages(pos, UNEVEN.lam_m, *_sky(seed), C, T, P, seed, device="cuda")
    s["vis"] = torch.empty((C, ne * (ne + 1) // 2, P, P, 2), dtype=torch.int32, device="cuda")
    s["img"] = torch.empty((C, 4 if P == 2 else 1, n, n), device="cuda")
    return s


def _run_corr_xfft(s):
    c = s["case"]
    hai.hai_correlate(_ctx(), s["volt"], c["channels"], c["samples"], c["elements"], c["pols"], s["vis"])
    hai.hai_xfft_image(_ctx(), s["layout"], s["vis"], c["channels"], s["img"])
    return {"vis": s["vis"], "img": s["img"]}


def _prepare_beamform(case, seed, s):
    S, C, T, P, N, K = (case[k] for k in ("stations", "channels", "samples", "pols", "elements", "beams"))
    s["volt"] = _noise((S, C, T, P, N, 2), seed)
    side = math.ceil(math.sqrt(K))
    w = I.bf_weights(_station(N)[0], UNEVEN.lam_m, _beam_dirs(side * side)[:K], P)
    s["w"] = torch.from_numpy(np.repeat(w[None], S, axis=0)).cuda()
    s["beams"] = torch.empty((S, C, T, K, P, 2), dtype=torch.int32 if case["shift"] < 0 else torch.int8, device="cuda")
    return s


def _run_beamform(s):
    c = s["case"]
    hai.hai_beamform(_ctx(), s["volt"], s["w"], c["stations"], c["channels"], c["samples"], c["beams"], c["elements"],
                     c["pols"], c["shift"], s["beams"])
    return s["beams"]


def _prepare_interstation(case, seed, s):
    S, K, C, T, n = (case[k] for k in ("stations", "beams", "channels", "samples", "grid"))
    lay = hai.hai_vis_layout_create(_ctx(), _centres(S), HIER.station.lam_m, HIER.cell_m, n, _beam_dirs(K))
    s["layout"] = s.own(lay, hai.hai_vis_layout_destroy)
    s["beams"] = _beams(case, seed, 0.03).permute(4, 1, 2, 0, 3, 5).contiguous()
    s["corr"] = torch.empty((K * C, T, 2, S, 2), dtype=torch.int8, device="cuda")
    s["vis"] = torch.empty((K * C, S * (S + 1) // 2, 2, 2, 2), dtype=torch.int32, device="cuda")
    s["img"] = torch.empty((K * C, 4, n, n), device="cuda")
    return s


def _run_interstation(s):
    c = s["case"]
    S, K, C, T = c["stations"], c["beams"], c["channels"], c["samples"]
    hai.hai_beams_to_corr(_ctx(), s["beams"], S, C, T, K, 2, s["corr"])
    hai.hai_correlate(_ctx(), s["corr"], K * C, T, S, 2, s["vis"])
    hai.hai_xfft_station_image(_ctx(), s["layout"], s["vis"], C, s["img"])
    return {"corr": s["corr"], "vis": s["vis"], "img": s["img"]}


def _prepare_xbf(case, seed, s):
    S, K, C, n = (case[k] for k in ("stations", "beams", "channels", "grid"))
    lay = hai.hai_xbf_layout_create(_ctx(), _centres(S), HIER.station.lam_m, HIER.cell_m, n, _beam_dirs(K),
                                    hai.HAI_XBF_OFFGRID_PAIRS, C, PREC[case["prec"]])
    s["layout"] = s.own(lay, hai.hai_xbf_layout_destroy)
    # visibilities of a 64-sample cadence, by a plain product of the beams
    v = torch.view_as_complex(_beams(dict(case, samples=64), seed, 0.03).float()).reshape(K * C, 64, 2 * S)
    full = torch.einsum("ctm,ctn->cmn", v, v.conj()).view(K * C, 2, S, 2, S)
    a, b = np.tril_indices(S)
    full = full[:, :, torch.from_numpy(a).cuda(), :, torch.from_numpy(b).cuda()]      # [pair][KC][p][q]
    s["vis"] = torch.view_as_real(full.permute(1, 0, 2, 3)).round().to(torch.int32).contiguous()
    s["img"] = torch.empty((K * C, 4, n, n), device="cuda")
    return s


def _run_xbf(s):
    hai.hai_xbf_station_image(_ctx(), s["layout"], s["vis"], s["case"]["channels"], s["img"])
    return s["img"]


def _prepare_fftcorr(case, seed, s):
    C, n, P = case["channels"], case["grid"], case["pols"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    s["img"] = torch.randn((C, 4 if P == 2 else 1, n, n), generator=gen, device="cuda")
    s["img"][:, :P] += 8.0                                        # the autos' noise floor
    s["grid"] = torch.empty((C, P, P, n, n, 2), device="cuda")
    return s


def _run_fftcorr(s):
    c = s["case"]
    hai.hai_fft_correlate(_ctx(), s["img"], c["channels"], c["grid"], c["pols"], s["grid"])
    return s["grid"]


def _prepare_plan(case, seed, s):
    S, C, T, K = case["stations"], case["channels"], case["samples"], case["beams"]
    sizes, centres = _uneven(S)
    lays = [hai.hai_layout_create(_ctx(), _station(n)[1], _station(n)[2], _station(n)[3], 2) for n in sizes]
    plan = s["plan"] = s.own(hai.hai_plan_create(_ctx(), lays, C, T), hai.hai_plan_destroy)
    for lay in lays:
        hai.hai_layout_destroy(lay)
    dirs = _beam_dirs(K)
    w, off = I.uneven_beam_weights(UNEVEN, [_station(n)[0] for n in sizes], dirs)
    vl = hai.hai_vis_layout_create(_ctx(), centres, UNEVEN.lam_m, UNEVEN.xfft_cell_m, UNEVEN.xfft_grid_n, dirs)
    s.own(vl, hai.hai_vis_layout_destroy)
    els = [hai.hai_station_epic_layout_create(_ctx(), centres, UNEVEN.lam_m, UNEVEN.epic_cell_m, UNEVEN.epic_grid_n,
                                              dirs, k)[0] for k in range(K)]
    for el in els:
        s.own(el, hai.hai_layout_destroy)
    hai.hai_plan_set_hierarchy(plan, K, torch.from_numpy(w).cuda(), off, UNEVEN.requant_shift, xfft=vl, epic=els)
    s["volt"] = _noise((64, (plan.volt_bytes + 63) // 64), seed).view(-1)[:plan.volt_bytes]
    nb, nv, nx, ne = hai.hai_plan_hier_sizes(plan)
    s["img"] = torch.empty(plan.img_floats, device="cuda")
    s["beams"] = torch.empty(nb, dtype=torch.int8, device="cuda")
    s["corr"] = torch.empty(nb, dtype=torch.int8, device="cuda")
    s["vis"] = torch.empty(nv, dtype=torch.int32, device="cuda")
    s["xfft_img"] = torch.empty(nx, device="cuda")
    s["epic_img"] = torch.empty(ne, device="cuda")
    return s


def _run_plan(s):
    names = ("img", "beams", "corr", "vis", "xfft_img", "epic_img")
    hai.hai_plan_run_hier(s["plan"], s["volt"], *[s[k] for k in names])
    return {k: s[k] for k in names}


_PREPARE = {"epic": _prepare_epic, "corr_xfft": _prepare_corr_xfft, "beamform": _prepare_beamform,
            "interstation": _prepare_interstation, "xbf": _prepare_xbf, "fftcorr": _prepare_fftcorr, "plan": _prepare_plan}
_RUN = {"epic": _run_epic, "corr_xfft": _run_corr_xfft, "beamform": _run_beamform, "interstation": _run_interstation,
        "xbf": _run_xbf, "fftcorr": _run_fftcorr, "plan": _run_plan}


# ------------------------------------------------------------------ work
def _epic_work(C, T, P, ne, k, n):
    """Voltages in, images out; gridding, one 2D FFT per field, squaring."""
    planes = 4 if P == 2 else 1
    return {"bytes": C * T * P * ne * 2 + C * planes * n * n * 4,
            "flops": C * T * P * (8.0 * ne * k * k + 5.0 * n * n * 2 * math.log2(n) + 8.0 * n * n)}


def _corr_work(C, T, P, ne):
    vis = C * (ne * (ne + 1) // 2) * P * P * 8
    return {"bytes": C * T * P * ne * 2 + vis, "flops": C * T * (ne * (ne + 1) // 2) * P * P * 8.0}


def _sum(*works):
    return {k: sum(w[k] for w in works) for k in ("bytes", "flops")}


def _image_work(C, planes, n):
    """Visibility grids to images: one 2D FFT for each pair of planes, the images written."""
    return {"bytes": C * planes * n * n * 4, "flops": C * planes / 2.0 * 5.0 * n * n * 2 * math.log2(n)}


def work(case):
    kind = case["kind"]
    C = case["channels"]
    if kind == "epic":
        if case["array"] == "disk":
            ne, k, n = case["elements"], 3, _station(case["elements"])[3]
        elif case["array"] == "lattice":
            ne, k, n = case["side"] ** 2, 1, _lattice(case["side"])[3]
        else:
            ne, k, n = case["elements"], 1, 128
        return _epic_work(C, case["samples"], case["pols"], ne, k, n)
    if kind == "corr_xfft":
        P, ne = case["pols"], case["elements"]
        return _sum(_corr_work(C, case["samples"], P, ne), _image_work(C, 4 if P == 2 else 1, _station(ne)[3]))
    if kind == "beamform":
        S, T, P, N, K = (case[k] for k in ("stations", "samples", "pols", "elements", "beams"))
        out = S * C * T * K * P * 2 * (4 if case["shift"] < 0 else 1)
        return {"bytes": S * C * T * P * N * 2 + S * K * P * N * 2 + out, "flops": 8.0 * S * C * T * P * N * K}
    if kind == "interstation":
        S, K, T, n = (case[k] for k in ("stations", "beams", "samples", "grid"))
        reorder = {"bytes": K * C * T * 2 * S * 2, "flops": 0.0}
        return _sum(reorder, _corr_work(K * C, T, 2, S), _image_work(K * C, 4, n))
    if kind == "xbf":
        S, K, n = case["stations"], case["beams"], case["grid"]
        pairs = len(_dropped_pairs(S, n)[0])
        return {"bytes": K * C * (pairs * 32 + 4 * n * n * 4), "flops": K * C * pairs * n * n * 16.0}
    if kind == "fftcorr":
        n, P = case["grid"], case["pols"]
        planes = 4 if P == 2 else 1
        return {"bytes": C * n * n * (planes * 4 + P * P * 8), "flops": C * planes / 2.0 * 5.0 * n * n * 2 * math.log2(n)}
    S, T, K = case["stations"], case["samples"], case["beams"]
    sizes, _ = _uneven(S)
    parts = [_epic_work(C, T, 2, n, 3, _station(n)[3]) for n in sizes]
    parts.append({"bytes": 2 * S * C * T * K * 4, "flops": sum(16.0 * C * T * n * K for n in sizes)})
    parts.append(_corr_work(K * C, T, 2, S))
    parts.append(_image_work(K * C, 4, UNEVEN.xfft_grid_n))
    parts.append(_epic_work(K * C, T, 2, S, 1, UNEVEN.epic_grid_n))
    return _sum(*parts)


# ------------------------------------------------------------------ 64-bit results
def _transform(grid):
    """sum_j (-1)^(jx+jy) g[j] exp(+2 pi i l.j / n) of [..., n, n]."""
    n = grid.shape[-1]
    sign = 1.0 - 2.0 * (torch.arange(n, device=grid.device) % 2)
    return torch.fft.ifft2(grid * (sign[:, None] * sign[None, :]), norm="forward")


def _epic_exact(volt, anchors, taps, n):
    """Images [C][Q][n][n] of int8 voltages [C][T][P][ne][2]; taps complex [ne][k][k], used conjugated."""
    C, T, P, ne, _ = volt.shape
    k = taps.shape[1]
    v, u = np.meshgrid(np.arange(k), np.arange(k), indexing="ij")
    cells = ((anchors[:, 1, None, None] + v) * n + anchors[:, 0, None, None] + u).reshape(ne, k * k)
    cells = torch.from_numpy(cells.astype(np.int64)).cuda()
    w = torch.from_numpy(np.conj(taps).reshape(ne, k * k).astype(np.complex128)).cuda()
    img = torch.zeros((C, 4 if P == 2 else 1, n, n), dtype=torch.float64, device="cuda")
    step = max(1, (1 << 25) // (P * n * n))
    for c in range(C):
        for t in range(0, T, step):
            e = torch.view_as_complex(volt[c, t:t + step].double())
            g = torch.zeros((e.shape[0], P, n * n, 2), dtype=torch.float64, device="cuda")
            for q in range(k * k):
                g.index_add_(2, cells[:, q], torch.view_as_real(e * w[:, q]))
            f = _transform(torch.view_as_complex(g).view(-1, P, n, n))
            img[c, 0] += (f[:, 0].real ** 2 + f[:, 0].imag ** 2).sum(0)
            if P == 2:
                img[c, 1] += (f[:, 1].real ** 2 + f[:, 1].imag ** 2).sum(0)
                xy = (f[:, 0] * f[:, 1].conj()).sum(0)
                img[c, 2] += xy.real
                img[c, 3] += xy.imag
    return img


def _station_taps(pos, lam, cell, n, direction):
    """Nearest cells and FP64 steering weights of stations as elements; those outside the central half weigh 0."""
    cells = np.floor(pos / cell + n / 2.0 + 0.5).astype(np.int64)
    on = np.all((cells >= n // 4) & (cells < n - n // 4), axis=1)
    turns = (pos @ np.asarray(direction)) / lam
    w = np.where(on, np.exp(-2j * np.pi * turns), 0.0)
    return np.where(on[:, None], cells, n // 2), w.reshape(-1, 1, 1)


def _offgrid(pos, cell, n, a, b):
    """Pairs whose 2 x 2 footprint, or its mirror's, leaves [-n/2, n/2 - 1]^2."""
    d = (pos[a] - pos[b]) / cell
    bad = np.zeros(len(a), bool)
    for u in (np.floor(d), np.floor(-d)):
        bad |= np.any((u < -(n // 2)) | (u + 1 > n // 2 - 1), axis=1)
    return bad


@functools.lru_cache(maxsize=8)
def _dropped_pairs(S, n):
    a, b = np.tril_indices(S)
    bad = _offgrid(_centres(S), HIER.cell_m, n, a, b) & (a != b)
    return a[bad], b[bad]


def _visibilities(beams):
    """[C][S(S+1)/2][2][2] complex128 of [C][T][2][S][2]."""
    C, T, P, S, _ = beams.shape
    a, b = (torch.from_numpy(x).cuda() for x in np.tril_indices(S))
    out = torch.empty((C, len(a), P, P), dtype=torch.complex128, device="cuda")
    for c in range(C):
        v = torch.view_as_complex(beams[c].double()).reshape(T, P * S)
        full = (v.T @ v.conj()).view(P, S, P, S)
        out[c] = full[:, a, :, b]
    return out


def _station_xfft_exact(beams, pos, lam, cell, n, dirs):
    """[K][C][4][n][n] of [K][C][T][2][S][2]."""
    K, C = beams.shape[:2]
    a, b = np.tril_indices(len(pos))
    keep = ~_offgrid(pos, cell, n, a, b)
    d = pos[a] - pos[b]
    img = torch.empty((K, C, 4, n, n), dtype=torch.float64, device="cuda")
    for k in range(K):
        vis = _visibilities(beams[k])[:, torch.from_numpy(keep).cuda()]
        ph = np.exp(2j * np.pi * np.mod(d[keep] @ dirs[k] / lam, 1.0))
        g = torch.zeros((C, 4, n * n, 2), dtype=torch.float64, device="cuda")
        for mirror in (False, True):
            uv = (-d[keep] if mirror else d[keep]) / cell
            u0 = np.floor(uv).astype(np.int64)
            f = uv - u0
            x = vis * torch.from_numpy(ph).cuda()[:, None, None]
            if mirror:
                x = x.conj().transpose(2, 3) * torch.from_numpy((a != b)[keep]).cuda()[:, None, None]
            x = torch.stack([x[:, :, 0, 0], x[:, :, 1, 1], x[:, :, 0, 1], torch.zeros_like(x[:, :, 0, 1])], dim=1)
            for t in range(4):
                w = np.where(t & 1, f[:, 0], 1 - f[:, 0]) * np.where(t >> 1, f[:, 1], 1 - f[:, 1])
                cell_of = np.mod(u0[:, 1] + (t >> 1), n) * n + np.mod(u0[:, 0] + (t & 1), n)
                g.index_add_(2, torch.from_numpy(cell_of).cuda(), torch.view_as_real(x * torch.from_numpy(w).cuda()))
        for c in range(C):
            o = _transform(torch.view_as_complex(g[c]).view(4, n, n))
            img[k, c] = torch.stack([o[0].real, o[1].real, o[2].real, o[2].imag])
    return img


def _xbf_exact(case, vis):
    """The direct sum over the dropped pairs and their mirrors, [K C][4][n][n]."""
    S, K, C, n = (case[k] for k in ("stations", "beams", "channels", "grid"))
    pos, lam, cell, dirs = _centres(S), HIER.station.lam_m, HIER.cell_m, _beam_dirs(K)
    a, b = _dropped_pairs(S, n)
    d = pos[a] - pos[b]
    v = torch.view_as_complex(vis[:, torch.from_numpy(a * (a + 1) // 2 + b).cuda()].double()).view(K, C, -1, 2, 2)
    steer = torch.from_numpy(np.exp(2j * np.pi * np.mod(dirs @ d.T / lam, 1.0))).cuda()
    v = v * steer[:, None, :, None, None]
    img = torch.zeros((K * C, 4, n * n), dtype=torch.float64, device="cuda")
    pix = torch.arange(n, device="cuda", dtype=torch.float64) - n // 2
    step = 256
    for i in range(0, len(a), step):
        dd = torch.from_numpy(d[i:i + step] / (n * cell)).cuda()
        turns = torch.remainder(pix[None, :, None] * dd[:, 1, None, None] + pix[None, None, :] * dd[:, 0, None, None], 1.0)
        phi = torch.polar(torch.ones_like(turns), 2 * math.pi * turns).view(-1, n * n)
        phi = torch.cat([phi.real, phi.imag])                                          # [2 pairs][pixels]
        x = v[:, :, i:i + step].reshape(K * C, -1, 2, 2)
        rows = []
        for p, q in ((0, 0), (1, 1)):
            rows.append(torch.cat([2 * x[:, :, p, q].real, -2 * x[:, :, p, q].imag], dim=1))
        s, m = x[:, :, 0, 1], x[:, :, 1, 0].conj()                                     # the pair and its mirror
        rows.append(torch.cat([(s + m).real, (m - s).imag], dim=1))
        rows.append(torch.cat([(s + m).imag, (s - m).real], dim=1))
        img += (torch.stack(rows, dim=1).view(K * C * 4, -1) @ phi).view(K * C, 4, n * n)
    return img.view(K * C, 4, n, n)


def _fftcorr_exact(img, P):
    C, _, n, _ = img.shape
    x = img.double()
    pairs = [x[:, 0].to(torch.complex128)]
    if P == 2:
        xy = torch.complex(x[:, 2], x[:, 3])
        pairs += [xy, xy.conj(), x[:, 1].to(torch.complex128)]
    sign = 1.0 - 2.0 * (torch.arange(n, device="cuda") % 2)
    g = torch.stack([torch.fft.fft2(p) / (n * n) * (sign[:, None] * sign[None, :]) for p in pairs], dim=1)
    return torch.view_as_real(g.view(C, P, P, n, n))


def exact(case, seed):
    kind = case["kind"]
    if kind == "beamform":
        return None                                     # whole numbers
    if kind == "epic":
        if case["array"] == "stations":
            pos = _centres(case["elements"])
            anchors, taps = _station_taps(pos, HIER.station.lam_m, HIER.cell_m, 128, _beam_dirs(16)[5])
            return _epic_exact(_beams(case, seed, 0.03)[0], anchors, taps, 128)
        lat = case["array"] == "lattice"
        pos, anchors, taps, n = _lattice(case["side"]) if lat else _station(case["elements"])
        volt = I.voltages(pos, I.DENSE_ALLSKY_16384.lam_m if lat else UNEVEN.lam_m, *_sky(seed), case["channels"],
                          case["samples"], case["pols"], seed, device="cuda")
        return _epic_exact(volt, anchors, taps[..., 0] + 1j * taps[..., 1].astype(np.float64), n)
    if kind == "corr_xfft":                             # the same image as the direct imager's
        pos, anchors, taps, n = _station(case["elements"])
        volt = I.voltages(pos, UNEVEN.lam_m, *_sky(seed), case["channels"], case["samples"], case["pols"], seed,
                          device="cuda")
        return {"vis": None, "img": _epic_exact(volt, anchors, taps[..., 0].astype(np.complex128), n)}
    if kind == "interstation":
        S, n = case["stations"], case["grid"]
        img = _station_xfft_exact(_beams(case, seed, 0.03), _centres(S), HIER.station.lam_m, HIER.cell_m, n,
                                  _beam_dirs(case["beams"]))
        return {"corr": None, "vis": None, "img": img.view(-1, 4, n, n)}
    if kind == "xbf":
        return _xbf_exact(case, prepare(case, seed)["vis"])
    if kind == "fftcorr":
        return _fftcorr_exact(prepare(case, seed)["img"], case["pols"])
    # the plan: station images; the second level's from the requantised beams
    s = prepare(case, seed)
    S, C, T, K = case["stations"], case["channels"], case["samples"], case["beams"]
    sizes, centres = _uneven(S)
    dirs, lam = _beam_dirs(K), UNEVEN.lam_m
    beams = torch.empty((K, C, T, 2, S, 2), dtype=torch.int8, device="cuda")
    img = torch.empty(s["plan"].img_floats, dtype=torch.float64, device="cuda")
    half = 1 << (UNEVEN.requant_shift - 1)
    for i, ne in enumerate(sizes):
        pos, anchors, taps, n = _station(ne)
        o = int(s["plan"].volt_off[i])
        v = s["volt"][o:o + C * T * 2 * ne * 2].view(C, T, 2, ne, 2)
        o = int(s["plan"].img_off[i])
        img[o:o + C * 4 * n * n] = _epic_exact(v, anchors, taps[..., 0].astype(np.complex128), n).view(-1)
        w = torch.view_as_complex(torch.from_numpy(I.bf_weights(pos, lam, dirs, 2)).cuda().double())   # [K][2][ne]
        b = torch.view_as_real(torch.einsum("kpn,ctpn->kctp", w.conj(), torch.view_as_complex(v.double()))).round()
        b = torch.sign(b) * torch.floor((b.abs() + half) / (2 * half))
        beams[:, :, :, :, i] = b.clamp(-127, 127).to(torch.int8)
    xfft = _station_xfft_exact(beams, centres, lam, UNEVEN.xfft_cell_m, UNEVEN.xfft_grid_n, dirs)
    epic = []
    for k in range(K):
        anchors, taps = _station_taps(centres, lam, UNEVEN.epic_cell_m, UNEVEN.epic_grid_n, dirs[k])
        epic.append(_epic_exact(beams[k], anchors, taps, UNEVEN.epic_grid_n))
    return {"img": img, "beams": None, "corr": None, "vis": None, "xfft_img": xfft.view(-1),
            "epic_img": torch.stack(epic).view(-1)}
