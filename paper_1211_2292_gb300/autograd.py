"""Differentiable leapfrog rollout over the library's adjoint kernels.

``rollout(nb, x0, v0, m, G, eps, dt, nsteps, every)`` runs ``nsteps``
kick-drift-kick steps (the reading of the paper's "Move_bodies", Sec. IV-B)
and returns the final positions and velocities as tensors that torch
autograd can differentiate with respect to x0, v0 and m.

Forward: one ``nb_rollout`` call that records the state every ``every``
steps (segment checkpoints).  Backward, segment by segment from the last:
restore the checkpoint, recompute the positions up to the next checkpoint with
``nb_rollout(record_every=1)``, which ends after the last of them is reached
(``NB_END_AT_DRIFT``), then run ``nb_step_backward`` (the reverse sweep with the
force VJP kernel).  Memory:
(nsteps/every + 1) checkpoints of (x, v) plus one segment of positions;
compute: every - 1 force evaluations per segment of `every` steps.  (With the
segment's end position and the force there computed again too, every + 1:
2.63 ms for 4 steps of 16384 bodies with every = 2, 2.30 now.  Three torch operations
per segment in the place of ``NB_END_AT_DRIFT`` made a small system's backward, which
is the host's, 12 % longer: 735 us for 4 steps of 300 bodies, 670 now.)

Library calls and torch operations meet on the context's stream, whichever
stream the caller is on (``NBody.in_order``): the tensors are allocated on the
caller's stream, which waits for the context's before it goes on.
"""
from __future__ import annotations

import torch

from .nbody import NBody


class NBodyRollout(torch.autograd.Function):
    @staticmethod
    def forward(ctx, x0, v0, m, nb: NBody, G: float, eps: float, dt: float, nsteps: int,
                every: int):
        every = max(1, int(every))
        nsteps = int(nsteps)
        n = m.shape[0]
        x = torch.empty_like(x0).copy_(x0.detach())
        v = torch.empty_like(v0).copy_(v0.detach())
        md = m.detach().contiguous()
        acc = torch.empty_like(x)
        nrec = nsteps // every + 1
        ckx = torch.empty((nrec, n, 3), dtype=x.dtype, device=x.device)
        ckv = torch.empty_like(ckx)
        if nsteps > 0:
            with nb.in_order():
                nb.rollout(x, v, md, G, eps, dt, nsteps, acc, every, ckx, ckv)
        ctx.nb, ctx.G, ctx.eps, ctx.dt, ctx.nsteps, ctx.every = nb, G, eps, dt, nsteps, every
        ctx.save_for_backward(ckx, ckv, md)
        return x, v

    @staticmethod
    def backward(ctx, gx, gv):
        ckx, ckv, m = ctx.saved_tensors
        nb, G, eps, dt, nsteps, every = ctx.nb, ctx.G, ctx.eps, ctx.dt, ctx.nsteps, ctx.every
        n = m.shape[0]
        lam_x = torch.zeros((n, 3), dtype=m.dtype, device=m.device)
        lam_v = torch.zeros_like(lam_x)
        if gx is not None:
            lam_x.copy_(gx)
        if gv is not None:
            lam_v.copy_(gv)
        lam_m = torch.zeros_like(m)
        if nsteps == 0:
            return lam_x, lam_v, lam_m, None, None, None, None, None, None
        nseg = (nsteps + every - 1) // every
        if every == 1:
            traj = ckx.to(m).contiguous()  # (as a hook may have unpacked it)
        else:
            traj = torch.empty((every + 1, n, 3), dtype=m.dtype, device=m.device)
            x = torch.empty((n, 3), dtype=m.dtype, device=m.device)
            v, acc = torch.empty_like(x), torch.empty_like(x)
            xs, vs, upto, end = ckx.unbind(0), ckv.unbind(0), traj[:every], traj[every]
        with nb.in_order():  # the loop's own torch operations too
            for s in range(nseg - 1, -1, -1):
                start = s * every
                length = min(every, nsteps - start)
                if every == 1:
                    seg = traj[s: s + 2]
                else:
                    # the positions after the first are computed again, but for the
                    # last of a whole segment: that one is the next checkpoint
                    x.copy_(xs[s])
                    v.copy_(vs[s])
                    if length == every:
                        seg, rec, new = traj, upto, every - 1
                        end.copy_(xs[s + 1])
                    else:
                        seg = rec = traj[: length + 1]
                        new = length
                    nb.rollout(x, v, m, G, eps, dt, new, acc, 1, rec, end_at_drift=True)
                nb.step_backward(seg, m, G, eps, dt, length, lam_x, lam_v, lam_m,
                                 at_start=(s == 0), at_end=(s == nseg - 1))
        return lam_x, lam_v, lam_m, None, None, None, None, None, None


def rollout(nb: NBody, x0, v0, m, G: float, eps: float, dt: float, nsteps: int, every: int = 20):
    """Final (x, v) after nsteps leapfrog steps, differentiable in (x0, v0, m)."""
    return NBodyRollout.apply(x0, v0, m, nb, G, eps, dt, nsteps, every)
