"""Autotuner for the persistent sweep grid.

Times short solves of the caller's own system under candidate launch
configurations and returns the fastest: the block shape of the cooperative
sweep grid (threads per block x blocks per SM).  Every candidate keeps the
Gauss-Seidel order, so choosing among them changes only the speed.

Everything runs through the CUDA library (``cd.CDSystem``); each trial is
timed with the CUDA events the library records around the sweep kernel.
"""
from __future__ import annotations

from . import cd

BLOCK_SHAPES = [(512, 1), (256, 2), (256, 1), (128, 4), (128, 2)]
ORDER_KEEPING = [dict(sweep_threads=t, sweep_blocks_per_sm=b) for t, b in BLOCK_SHAPES]


# Up to this cap cd_create_system solves a plain system behind barriers, above it
# (in the default block shape, where nothing else is asked for) by dataflow.
SHORT_SOLVE = 128
LONG_TRIAL = 160   # sweeps that are on the far side of it, and set-up a small part of them


def trial_sweeps(sweeps, cap):
    """Sweeps of a timed solve for a system capped at `cap`: `sweeps`, but by the
    kernel that the system will run.  (Trials of 40 sweeps timed the barrier
    kernel for systems whose solves run by dataflow, and for piles of up to
    20,000 discs chose 256 x 1, 2% faster there and half as fast as the
    dataflow of 512 x 1 that it switched off.)"""
    return min(sweeps, SHORT_SOLVE) if cap <= SHORT_SOLVE else max(sweeps, LONG_TRIAL)


def tune(wl, batch=None, precision=cd.CD_FP64, sweeps=40, steps=2, device="cuda", candidates=None,
         max_contacts=None, max_sweeps=None):
    """Returns (best parameter dict, table of (parameters, ms per sweep)).

    Each candidate system is built over the workload (or the batch), stepped
    once untimed, then `steps` steps of `sweeps` sweeps (`trial_sweeps`, for the
    cap `max_sweeps`, by default the workload's) are timed; the
    figure is the sweep kernel's device time per sweep.  Candidates the
    device or the system cannot run (a schedule a batch does not support, a
    shape that does not fit) are skipped."""
    cap = (batch[0] if batch else wl).max_sweeps if max_sweeps is None else max_sweeps
    sweeps = trial_sweeps(sweeps, cap)
    cands = list(candidates) if candidates is not None else list(ORDER_KEEPING)
    table = []
    for kw in cands:
        extra = dict(kw)
        if max_contacts is not None:
            extra["max_contacts"] = max_contacts
        try:
            g = cd.CDSystem(wl, device=device, batch=batch, precision=precision, criterion=cd.CD_CONV_NONE,
                            max_sweeps=sweeps, timing=1, **extra)
            g.step(1)
            st = g.step(steps)
        except cd.CDError:
            continue
        ms = st["phase_ms"]["sweep"] / (steps * max(st["last"]["sweeps"], 1))
        table.append((dict(kw), ms))
        del g
    if not table:
        raise RuntimeError("no candidate configuration could run")
    best = min(table, key=lambda t: t[1])[0]
    return best, table
