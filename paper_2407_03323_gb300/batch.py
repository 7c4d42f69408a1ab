"""Batched marching of many scatterers (uneven grids) x excitations on one GPU.

Each scatterer gets one context (the setup: element quadrature, spatial and level
spectra) and mot_create_shared contexts for its other excitations, so the setup is
computed once per scatterer.  All marches advance in lockstep chunks; every context is
driven from its own host thread (the library calls release the GIL), so the kernels of
different contexts run concurrently on their own streams.  With rhs=True a scatterer's
excitations are instead the right-hand sides of its one context
(mot_set_excitation_rhs / mot_march_rhs: one call interleaves their steps on their
streams) and the pool drives scatterers; measured slower when it was written (3.9e8 against 4.2e8
voxel-timesteps/s on the 24 x 8 workload, 5.4e8 now without it), so it is off by default.  Scatterers are processed in
waves whose march state fits a device-memory budget.  Each round first stages every
march's excitation chunk on the device (the tested plane wave, generated by the
library), then times the marches of the round; setup, tuning and excitation staging
are outside the march time.

Each march call covers one chunk; with `graphs` the library captures the chunk's
launches into a CUDA graph and replays it, updated in place, for the later chunks
(mot_set_graph), so a chunk costs one graph launch instead of ~10 launches per step.
Off by default: these marches are bound by the latency of the solve's iterations, not
by launches (a graph saves 2-3 % per step in steady state), and the capture, update
and first instantiation of every context's graph cost more host time than that over
a few hundred steps.

The block size B of the blocked history scheme is picked per scatterer by
`BlockTuner`: for each size bucket it times a short march (two periods of the longest
level) of every candidate B on a probe grid of the bucket's largest side and keeps the
fastest.  Argument marshalling only: every step runs in the library's kernels.
"""
import concurrent.futures
import time

import numpy as np
import torch

from .mot import Context, codelet_size, pad_size


def _state_bytes(N, precision, block, P=None):
    """Device bytes of one excitation's rings on an N^3 grid with FFT length P (default: the
    library's padding): spectral ring and far-level accumulators, the accumulators counted for
    the doubling level plan, an upper bound; with 200 bytes a voxel beside them."""
    P = P or pad_size(N)
    c = 8 if precision == "fp32_history" else 16
    slot = 3 * P * P * (P // 2 + 1) * c
    ell = int(np.floor(N * np.sqrt(3.0))) + 2
    acc, S = 0, block
    while block and S <= ell:
        acc += S
        S *= 2
    return slot * (ell + acc) + 200 * N ** 3


def march_bytes(N, precision, block, P=None, n_taps=3):
    """Device bytes of one excitation's whole march state: _state_bytes with what it leaves out,
    the product's spectrum, the transforms' intermediates and the rest of the solve's state.  Per
    voxel that is the J ring (24 a slot), the six fitted right-hand sides and the current one
    (168), rhs and lambda (48), the inner vectors (64) and the history (24, or 12 with 28 for the
    low parts of b and x)."""
    P = P or pad_size(N)
    f32 = precision == "fp32_history"
    c, Hu = 8 if f32 else 16, P // 2 + 1
    voxel = 24 * (max(n_taps, 6) + 1) + 168 + 48 + 64 + (40 if f32 else 24)
    planes = 3 * P * P * Hu * c + 3 * N * (N + P) * Hu * c
    return _state_bytes(N, precision, block, P) + planes + (voxel - 200) * N ** 3 + (1 << 20)


def fft_lengths(N, strategy):
    """Zero-padded FFT length of an N^3 grid per axis: the smallest even 7-smooth length
    >= 2N - 1 ('pad'), or the smallest length with a four-step codelet when it is at
    most 1.5 times that ('codelet')."""
    P = pad_size(N) if strategy == "pad" else codelet_size(N)
    return (P, P, P)


class BlockTuner:
    """Pick the blocked scheme's block length B (the lag-block schedule: near lags below
    B, far levels from B on) and the FFT length strategy (the radix plan: smallest
    7-smooth length or a length with a four-step codelet) by timing the candidates on
    probe grids of each size bucket (cached)."""

    def __init__(self, precision="fp32_history", candidates=(4, 8, 16), buckets=(24, 32, 40, 48),
                 strategies=("pad", "codelet")):
        self.precision = precision
        self.candidates = candidates
        self.buckets = buckets
        self.strategies = strategies
        self.choice = {}
        self.timings = {}

    def bucket(self, N):
        for b in self.buckets:
            if N <= b:
                return b
        return N

    def _tune(self, b):
        eps = np.full((b, b, b), 12.0)
        best = None
        strategies = [st for st in self.strategies
                      if st == "pad" or fft_lengths(b, st) != fft_lengths(b, "pad")]
        for st in strategies:
            for B in self.candidates:
                with Context(eps, [0.25e-7 * b ** 3, -0.5e-7 * b ** 3, 0.25e-7 * b ** 3],
                             precision=self.precision, scheme="blocked", block=B,
                             fft_len=fft_lengths(b, st)) as ctx:
                    if not ctx.levels:
                        continue
                    n = 2 * ctx.period
                    ctx.march(ctx.period, out=None)              # warm-up period
                    t0 = time.perf_counter()
                    ctx.march(n, out=None)
                    dt = (time.perf_counter() - t0) / n
                key = (b, B) if st == "pad" else (b, B, st)
                self.timings[key] = dt
                if best is None or dt < best[2]:
                    best = (B, st, dt)
        self.choice[b] = best[:2]

    def __call__(self, N):
        """Block length B for an N^3 grid."""
        b = self.bucket(N)
        if b not in self.choice:
            self._tune(b)
        return self.choice[b][0]

    def fft_len(self, N):
        """FFT lengths for an N^3 grid under its bucket's chosen strategy."""
        b = self.bucket(N)
        if b not in self.choice:
            self._tune(b)
        return fft_lengths(N, self.choice[b][1])


def _stage_chunk(ctx, wave, n_first, n, Ebuf):
    """Tested excitation of steps n_first .. n_first + n - 1, staged on the device."""
    E = Ebuf[:n]
    ctx.plane_wave(wave["k_hat"], wave["p_hat"], wave["f_c"], wave["sigma_t"], wave["t0"],
                   n_first, n, out=E)
    ctx.set_excitation(E)


def _march_chunk(ctx, n):
    ctx.march(n, out=None)
    return ctx.info()["last_norm"]


def _stage_rhs(ctx, waves, n_first, n, Ebuf):
    """Tested excitations of every right-hand side for steps n_first .. n_first + n - 1,
    staged on the device (mot_set_excitation_rhs)."""
    # the right-hand sides' steps contiguous ([r][n][M][3]): a shorter last chunk gets
    # its own buffer rather than a strided view of the chunk buffer
    E = Ebuf if n == Ebuf.shape[1] else torch.empty((Ebuf.shape[0], n) + tuple(Ebuf.shape[2:]),
                                                      dtype=Ebuf.dtype, device=Ebuf.device)
    for r, w in enumerate(waves):
        ctx.plane_wave(w["k_hat"], w["p_hat"], w["f_c"], w["sigma_t"], w["t0"], n_first, n,
                       out=E[r])
    ctx.set_excitation_rhs(E)


def _march_rhs_chunk(ctx, n_rhs, n):
    ctx.march_rhs(n, out=None)
    return [ctx.rhs(r).info()["last_norm"] for r in range(n_rhs)]


def run_batched(instances, n_steps, precision="fp32_history", tuner=None, chunk=64,
                memory_budget=120e9, workers=8, graphs=False, rhs=False):
    """March every (scatterer, excitation) of `instances` (workloads.batched_instances)
    for n_steps.  Returns timing, the aggregate voxel-timesteps/s of the marches and the
    chosen block sizes; setup and tuning are excluded from the march time.  graphs:
    march whole chunks as CUDA graphs (mot_set_graph with one chunk per graph, where the
    chunk is a whole number of the context's longest level period).  rhs: one context
    per scatterer carries all its excitations (mot_set_excitation_rhs / mot_march_rhs:
    the steps of its right-hand sides interleaved on their streams by one call);
    otherwise every excitation is a context of its own (mot_create_shared) marched by
    its own call."""
    tuner = tuner or BlockTuner(precision)
    blocks = [tuner(inst["N"]) for inst in instances]
    order = sorted(range(len(instances)), key=lambda i: -instances[i]["N"])
    waves, cur, used = [], [], 0.0
    for i in order:
        need = len(instances[i]["waves"]) * march_bytes(instances[i]["N"], precision, blocks[i],
                                                         tuner.fft_len(instances[i]["N"])[0],
                                                         len(instances[i]["taps"]))
        if cur and used + need > memory_budget:
            waves.append(cur)
            cur, used = [], 0.0
        cur.append(i)
        used += need
    if cur:
        waves.append(cur)
    march_s = setup_s = 0.0
    voxel_steps = 0
    last_norms = {}
    pool = concurrent.futures.ThreadPoolExecutor(max_workers=workers)
    try:
        for wave_ids in waves:
            if rhs:
                t0 = time.perf_counter()
                groups = []                             # (ctx, waves, E buffer, i)
                for i in wave_ids:
                    inst = instances[i]
                    src = Context(inst["eps_r"], inst["taps"], precision=precision,
                                  scheme="blocked", block=blocks[i],
                                  fft_len=tuner.fft_len(inst["N"]))
                    E = torch.empty((len(inst["waves"]), chunk, src.M, 3), dtype=torch.float64,
                                    device="cuda")
                    groups.append((src, inst["waves"], E, i))
                torch.cuda.synchronize()
                setup_s += time.perf_counter() - t0
                done = 0
                while done < n_steps:
                    k = min(chunk, n_steps - done)
                    for c, ws, E, _ in groups:
                        _stage_rhs(c, ws, done + 1, k, E)
                    torch.cuda.synchronize()
                    t0 = time.perf_counter()
                    futs = [pool.submit(_march_rhs_chunk, c, len(ws), k) for c, ws, _, _ in groups]
                    for f, (_, _, _, i) in zip(futs, groups):
                        for j, v in enumerate(f.result()):
                            last_norms[(i, j)] = v
                    torch.cuda.synchronize()
                    march_s += time.perf_counter() - t0
                    done += k
                voxel_steps += sum(c.M * len(ws) for c, ws, _, _ in groups) * n_steps
                for c, _, _, _ in groups:
                    c.close()
                del groups
                torch.cuda.empty_cache()
                continue
            t0 = time.perf_counter()
            runs = []                                   # (ctx, wave, E buffer, key)
            owners = []
            for i in wave_ids:
                inst = instances[i]
                src = Context(inst["eps_r"], inst["taps"], precision=precision,
                              scheme="blocked", block=blocks[i], fft_len=tuner.fft_len(inst["N"]))
                owners.append(src)
                ctxs = [src] + [src.share() for _ in inst["waves"][1:]]
                for j, (c, w) in enumerate(zip(ctxs, inst["waves"])):
                    if graphs and chunk % c.period == 0:
                        c.set_graph(chunk)
                    E = torch.empty((chunk, c.M, 3), dtype=torch.float64, device="cuda")
                    runs.append((c, w, E, (i, j)))
            torch.cuda.synchronize()
            setup_s += time.perf_counter() - t0
            done = 0
            while done < n_steps:
                k = min(chunk, n_steps - done)
                # inputs of the round resident on the device before its timed region
                for c, w, E, _ in runs:
                    _stage_chunk(c, w, done + 1, k, E)
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                futs = [pool.submit(_march_chunk, c, k) for c, _, _, _ in runs]
                for f, (_, _, _, key) in zip(futs, runs):
                    last_norms[key] = f.result()
                torch.cuda.synchronize()
                march_s += time.perf_counter() - t0
                done += k
            voxel_steps += sum(c.M for c, _, _, _ in runs) * n_steps
            for c, _, _, _ in runs:
                if c not in owners:
                    c.close()
            for c in owners:
                c.close()
            del runs
            torch.cuda.empty_cache()
    finally:
        pool.shutdown()
    return {"march_s": march_s, "setup_s": setup_s, "voxel_steps": voxel_steps,
            "value": voxel_steps / march_s, "blocks": blocks, "waves": len(waves),
            "fft_lengths": [tuner.fft_len(inst["N"])[0] for inst in instances],
            "tuning": {("%d/B=%d" % k[:2]) + ("/" + k[2] if len(k) > 2 else ""): v
                       for k, v in tuner.timings.items()},
            "last_norms": last_norms}
