"""Solver: one IDUGKS problem on one GPU through the C ABI.

PyTorch only provides the device workspace and the CUDA stream; every step of
the scheme runs in libidugks.
"""
from __future__ import annotations

import numpy as np

from . import binding as B
from .inputs import Problem, with_params


def configure(ctx, prob: Problem, explicit: bool = False):
    """Pass a Problem description to a fresh context (setters of include/idugks.h).
    explicit: the context advances explicit DUGKS steps (IDG_NUM_EXPLICIT)."""
    if prob.flags:
        raise ValueError("Problem.flags selects oracle-only options; the library takes none")
    if prob.unstructured:
        B.idg_set_mesh_unstructured(ctx, prob.nodes_x, prob.nodes_y, prob.cell_nodes, prob.edge_side)
    else:
        B.idg_set_mesh_structured(ctx, prob.nodes_x, prob.nodes_y)
    x0, x1, y0, y1 = prob.vrange
    B.idg_set_velocity_grid(ctx, prob.vrule, prob.nvx, prob.nvy, x0, x1, y0, y1)
    B.idg_set_gas(ctx, prob.K, prob.Pr, prob.omega, prob.Kn, prob.RT_ref,
                  B.IDG_SHAKHOV if prob.shakhov else B.IDG_BGK)
    for side in range(4):
        kind, rho, u, v, T = prob.bc[side]
        B.idg_set_boundary(ctx, side, kind, rho, u, v, T)
    B.idg_set_numerics(ctx, prob.cfl_imp, prob.cfl_phys, prob.limiter, prob.lusgs_omega,
                       B.IDG_NUM_EXPLICIT if explicit else 0)
    if prob.relax_sweeps:
        B.idg_set_predictor(ctx, prob.relax_sweeps)
    if getattr(prob, "implicit_wall", 0):
        B.idg_set_implicit_wall(ctx, 1)
    if getattr(prob, "venkat_k", 0.0):
        B.idg_set_limiter_smoothing(ctx, prob.venkat_k)


class Solver:
    """IDUGKS steady solver for one Problem.

    precision: "fp64" (f in float64) or "mixed" (f in float32, moments,
    macroscopic predictor and residual in float64).
    explicit: iterate() advances explicit DUGKS time steps (Eq. 21) instead of
    IDUGKS iterations.
    """

    def __init__(self, prob: Problem, precision: str = "fp64", device: int = 0, stream=None,
                 explicit: bool = False):
        import torch

        self.prob = prob
        self.device = device
        self.torch = torch
        p = B.IDG_FP64 if precision == "fp64" else B.IDG_MIXED
        self.precision = precision
        self.ctx = B.idg_create(p, device)
        self.explicit = explicit
        configure(self.ctx, prob, explicit)
        self.N, self.Nv, self.nf = B.idg_get_sizes(self.ctx)
        nbytes = B.idg_workspace_size(self.ctx)
        self.workspace = torch.empty(nbytes + 256, dtype=torch.uint8, device=f"cuda:{device}")
        base = self.workspace.data_ptr()
        aligned = (base + 255) & ~255
        self._stream = stream
        B.idg_bind_workspace(self.ctx, aligned, nbytes)

    @property
    def stream(self):
        if self._stream is not None:
            return self._stream
        return self.torch.cuda.current_stream(self.device).cuda_stream

    def __del__(self):
        ctx = getattr(self, "ctx", None)
        if ctx is not None:
            B.idg_destroy(ctx)
            self.ctx = None

    @property
    def dt(self) -> float:
        return B.idg_get_dt(self.ctx)

    def velocity_grid(self):
        return B.idg_velocity_grid(self.ctx, self.Nv)

    def init_uniform(self, rho=None, u=None, v=None, T=None):
        r0, u0, v0, T0 = self.prob.init
        B.idg_init_uniform(self.ctx, r0 if rho is None else rho, u0 if u is None else u,
                           v0 if v is None else v, T0 if T is None else T, self.stream)

    def set_state(self, G, H, W):
        B.idg_set_state(self.ctx, G, H, W, self.stream)

    def get_state(self):
        return B.idg_get_state(self.ctx, self.N, self.Nv, self.stream)

    def save(self, path):
        """Checkpoint the state to a file (idg_save)."""
        B.idg_save(self.ctx, path, self.stream)

    def load(self, path):
        """Restart from a checkpoint file (idg_load)."""
        B.idg_load(self.ctx, path, self.stream)

    def iterate(self, max_iter: int, tol: float = 0.0):
        """Returns (converged, iterations, relative residual)."""
        st, n, r = B.idg_iterate(self.ctx, max_iter, tol, self.stream)
        return st == B.IDG_OK, n, r

    def iterate_profiled(self) -> np.ndarray:
        """One iteration; device ms of cell prep, reconstruction with the face moments,
        face flux, macroscopic predictor, micro residual with the forward sweep,
        backward sweep."""
        return B.idg_iterate_profiled(self.ctx, self.stream)

    def set_tuning(self, **kw):
        """sweep_tv=, sweep_vpt=, sweep_stages=, macro_stages=, macro_kind=, graph=
        (launch shapes only)."""
        keys = {"sweep_tv": B.IDG_TUNE_SWEEP_TV, "sweep_stages": B.IDG_TUNE_SWEEP_STAGES,
                "macro_stages": B.IDG_TUNE_MACRO_STAGES, "graph": B.IDG_TUNE_GRAPH,
                "sweep_vpt": B.IDG_TUNE_SWEEP_VPT, "macro_kind": B.IDG_TUNE_MACRO_KIND}
        # only the given keys are set: the untouched ones keep the library's own choice.
        # A shallower prefetch comes first, and a wider tile with one velocity per thread,
        # so that it fits on the way
        if "sweep_stages" in kw and int(kw["sweep_stages"]) <= B.idg_get_tuning(self.ctx, keys["sweep_stages"]):
            B.idg_set_tuning(self.ctx, keys["sweep_stages"], int(kw["sweep_stages"]))
        if "sweep_tv" in kw and "sweep_vpt" in kw:
            B.idg_set_tuning(self.ctx, keys["sweep_vpt"], 1)
        # (a macro_kind re-derives the macroscopic depth: macro_stages comes after it)
        for k in ("graph", "macro_kind", "sweep_tv", "sweep_vpt", "sweep_stages", "macro_stages"):
            if k in kw:
                B.idg_set_tuning(self.ctx, keys[k], int(kw[k]))

    def tuning(self) -> dict:
        return {"sweep_tv": B.idg_get_tuning(self.ctx, B.IDG_TUNE_SWEEP_TV),
                "sweep_stages": B.idg_get_tuning(self.ctx, B.IDG_TUNE_SWEEP_STAGES),
                "macro_stages": B.idg_get_tuning(self.ctx, B.IDG_TUNE_MACRO_STAGES),
                "graph": B.idg_get_tuning(self.ctx, B.IDG_TUNE_GRAPH),
                "sweep_vpt": B.idg_get_tuning(self.ctx, B.IDG_TUNE_SWEEP_VPT),
                "macro_kind": B.idg_get_tuning(self.ctx, B.IDG_TUNE_MACRO_KIND)}

    def moments(self) -> np.ndarray:
        return B.idg_get_moments(self.ctx, self.N, self.stream)

    def residual_history(self) -> np.ndarray:
        return B.idg_get_residual_history(self.ctx, 1 << 20)

    def face_flux_moments(self) -> np.ndarray:
        return B.idg_get_face_flux_moments(self.ctx, self.nf, self.stream)

    def wall_force(self, side_mask: int) -> np.ndarray:
        """(Fx, Fy) of the gas on the walls of the sides in side_mask, from the
        face fluxes of the last iteration."""
        return B.idg_get_wall_force(self.ctx, side_mask, self.stream)

    def wall(self, side: int) -> np.ndarray:
        """Per face of a wall side, from the last iteration: midpoint x, y, pressure
        p, shear stress tau_w and heat flux into the wall q_n ([nface][5])."""
        return B.idg_get_wall(self.ctx, side, self.stream)

    def adjoint(self, objective: int, side_mask: int, params, max_iter: int = 20000, tol: float = 1e-10,
                keep_state: bool = False, solver: str = "fixed_point", restart: int = 20,
                limiter: str = "exact"):
        """Discrete adjoint at the current state (idg_adjoint).  Returns
        (converged, J, dJ/dparams, iterations, relative update); with
        keep_state the adjoint variables stay readable by adjoint_state().
        solver: "fixed_point" (the transposed iteration) or "gmres" (restarted
        GMRES on the same linear system, domains with a far field).
        limiter: "exact" (the limiter factor differentiated) or "frozen" (held
        at the converged state: an approximate gradient, idg_set_adjoint_limiter)."""
        B.idg_set_adjoint_solver(self.ctx, B.IDG_ADJ_GMRES if solver == "gmres" else B.IDG_ADJ_FIXED_POINT,
                                 restart)
        B.idg_set_adjoint_limiter(self.ctx, B.IDG_ADJ_LIMITER_FROZEN if limiter == "frozen"
                                  else B.IDG_ADJ_LIMITER_EXACT)
        nbytes = B.idg_adjoint_workspace_size(self.ctx)
        ws = self.torch.empty(nbytes + 256, dtype=self.torch.uint8, device=f"cuda:{self.device}")
        aligned = (ws.data_ptr() + 255) & ~255
        st, J, g, n, r = B.idg_adjoint(self.ctx, objective, side_mask, list(params), aligned, nbytes,
                                       max_iter, tol, self.stream)
        self._adj_ws = (ws, aligned) if keep_state else None
        return st == B.IDG_OK, J, g, n, r

    def adjoint_state(self, which: int = 0):
        """(lambda_G, lambda_H, lambda_W) of the last adjoint(keep_state=True):
        which = 0 the adjoint of the gradient, 1 the objective's solve, 2 the
        total-mass solve of a closed domain."""
        ws, aligned = self._adj_ws
        return B.idg_adjoint_state(self.ctx, aligned, which, self.N, self.Nv, self.stream)


def apply_params(prob: Problem, params, values) -> Problem:
    """A copy of prob with the adjoint parameters (IDG_PARAM ids) set to values."""
    return with_params(prob, params, values)


class SteadySolve:
    """Differentiable steady solve: theta -> J, the force of the gas on walls.

    ``SteadySolve.apply(theta, spec)`` with theta a float64 tensor of the
    parameter values (spec.params, IDG_PARAM ids: wall temperature, wall
    velocity, Kn) converges the IDUGKS problem spec.problem with those values
    and returns J (a 0-d float64 tensor).  Its backward runs the hand-written
    discrete adjoint of libidugks (idg_adjoint) on the converged state; no
    iteration history is stored.  Built lazily on torch.autograd.Function.
    """

    _fn = None

    @classmethod
    def apply(cls, theta, spec: "SteadySpec"):
        if cls._fn is None:
            cls._fn = _make_steady_fn()
        return cls._fn.apply(theta, spec)


class NotConvergedError(RuntimeError):
    """A steady solve or its adjoint stopped at max_iter above its tolerance."""


class SteadySpec:
    """What SteadySolve solves.  strict (default True): a forward solve that
    does not reach tol, or an adjoint that does not reach adj_tol, raises
    NotConvergedError instead of returning J or a gradient of an unconverged
    state; with strict=False it warns and spec.last records the flags."""

    def __init__(self, problem: Problem, params, objective=B.IDG_OBJ_FORCE_X, side_mask=1 << B.IDG_JMAX,
                 precision="fp64", max_iter=20000, tol=1e-12, adj_max_iter=20000, adj_tol=1e-10,
                 strict=True):
        self.problem, self.params = problem, list(params)
        self.objective, self.side_mask, self.precision = objective, side_mask, precision
        self.max_iter, self.tol, self.adj_max_iter, self.adj_tol = max_iter, tol, adj_max_iter, adj_tol
        self.strict = strict
        self.last = None  # (solver, forward info, adjoint info) of the last call


def _not_converged(spec: SteadySpec, what: str, n: int, r: float, tol: float):
    msg = f"{what} stopped after {n} iterations at relative residual {r:.3g} > tol {tol:.3g}"
    if spec.strict:
        raise NotConvergedError(msg)
    import warnings
    warnings.warn(msg, RuntimeWarning, stacklevel=3)


def _make_steady_fn():
    import torch

    class _SteadySolveFn(torch.autograd.Function):
        @staticmethod
        def forward(ctx, theta, spec):
            vals = theta.detach().cpu().double().numpy()
            solver = Solver(apply_params(spec.problem, spec.params, vals), spec.precision)
            solver.init_uniform()
            ok, n, r = solver.iterate(spec.max_iter, spec.tol)
            spec.last = {"solver": solver, "converged": ok, "iterations": n, "residual": r}
            if not ok:
                _not_converged(spec, "steady solve", n, r, spec.tol)
            force = solver.wall_force(spec.side_mask)
            J = float(force[0 if spec.objective == B.IDG_OBJ_FORCE_X else 1])
            ctx.solver, ctx.spec = solver, spec
            return torch.tensor(J, dtype=torch.float64, device=theta.device)

        @staticmethod
        def backward(ctx, gJ):
            spec = ctx.spec
            ok, J, g, n, r = ctx.solver.adjoint(spec.objective, spec.side_mask, spec.params,
                                                spec.adj_max_iter, spec.adj_tol)
            spec.last.update({"adj_converged": ok, "adj_J": J, "adj_iterations": n, "adj_residual": r})
            if not ok:
                _not_converged(spec, "adjoint", n, r, spec.adj_tol)
            grad = torch.as_tensor(np.asarray(g), dtype=torch.float64, device=gJ.device)
            return gJ * grad, None

    return _SteadySolveFn


class BatchSolver:
    """Many Problems advanced together: each kernel of an iteration is launched
    once over all instances (idg_batch_*).  Instances may differ in size, gas,
    boundaries and tuning; all use one precision on one device."""

    def __init__(self, problems, precision: str = "mixed", device: int = 0, autotune: bool = False,
                 tuning: dict = None):
        """tuning: launch-shape keys of Solver.set_tuning applied to every
        instance (instead of autotune)."""
        import torch

        self.torch = torch
        self.device = device
        self.solvers = [Solver(p, precision, device) for p in problems]
        for s in self.solvers:
            s.init_uniform()
            if tuning:
                s.set_tuning(**tuning)
        if autotune:
            # one batch shares the velocities-per-thread of its sweeps: tune
            # the largest instance first and keep its choice for the rest
            tuner = Autotuner()
            order = sorted(self.solvers, key=lambda s: -s.N * s.Nv)
            tuner.candidates_vpt = (tuner.tune(order[0])["sweep_vpt"],)
            for s in order[1:]:
                tuner.tune(s)
        self._make_batch()
        if autotune and len(self.solvers) > 1:
            self._tune_sweep_stages()

    def _tune_sweep_stages(self, candidates=(8, 4, 2), iters: int = 4):
        """The micro sweeps' prefetch depth of the whole batch, timed on the
        batch itself: one instance alone runs fewer sweep blocks than the SMs
        hold, where a deeper prefetch pays; a batch runs many waves of them,
        where the shared memory a shallower one frees buys resident blocks.
        The instances are back at their uniform start afterwards."""
        torch = self.torch
        best = None
        for st in candidates:
            try:
                for s in self.solvers:
                    s.set_tuning(sweep_stages=st)
            except B.IdgError:
                continue
            self._remake()
            self.iterate(2)
            a, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            stream = torch.cuda.current_stream(self.device)
            a.record(stream)
            self.iterate(iters)
            e.record(stream)
            torch.cuda.synchronize(self.device)
            ms = a.elapsed_time(e)
            if best is None or ms < best[0]:
                best = (ms, st)
        for s in self.solvers:
            if best is not None:
                s.set_tuning(sweep_stages=best[1])
            s.init_uniform()
        self._remake()

    def _remake(self):
        B.idg_batch_destroy(self.handle)
        self.handle = None
        self._make_batch()

    def _make_batch(self):
        # largest wavefront first: every batched kernel lays its blocks out in
        # the batch's instance order and the hardware dispatches them in
        # block order, so the micro sweeps' longest tiles (ni + nj - 1 steps)
        # start first and the shortest fill the last wave
        self._order = sorted(range(len(self.solvers)),
                             key=lambda i: -(self.solvers[i].prob.ni + self.solvers[i].prob.nj))
        self.handle = B.idg_batch_create([self.solvers[i].ctx for i in self._order])
        nbytes = B.idg_batch_workspace_size(self.handle)
        self.workspace = self.torch.empty(nbytes + 256, dtype=self.torch.uint8, device=f"cuda:{self.device}")
        aligned = (self.workspace.data_ptr() + 255) & ~255
        B.idg_batch_bind_workspace(self.handle, aligned, nbytes)

    @property
    def stream(self):
        return self.torch.cuda.current_stream(self.device).cuda_stream

    @property
    def cell_velocities(self) -> int:
        return sum(s.N * s.Nv for s in self.solvers)

    def iterate(self, max_iter: int, tol: float = 0.0):
        """Returns (all converged, iterations launched, largest relative residual, per-instance flags)."""
        st, n, r, conv = B.idg_batch_iterate(self.handle, len(self.solvers), max_iter, tol, self.stream)
        flags = [False] * len(conv)
        for j, i in enumerate(self._order):
            flags[i] = conv[j]
        return st == B.IDG_OK, n, r, flags

    def __del__(self):
        h = getattr(self, "handle", None)
        if h is not None:
            B.idg_batch_destroy(h)
            self.handle = None


class Autotuner:
    """Picks the micro-sweep tile (velocities per thread block and per thread)
    and the prefetch depths of a Solver by timing one profiled iteration of
    each candidate on the problem itself; results are cached per (cells in i,
    in j, velocities, precision) so a batch of same-sized problems is timed
    once."""

    def __init__(self, candidates_tv=(2, 4, 8, 16), candidates_vpt=(1, 2, 4), repeats: int = 3):
        self.candidates_tv = candidates_tv
        self.candidates_vpt = candidates_vpt
        self.repeats = repeats
        self.cache = {}

    def tune(self, solver: "Solver") -> dict:
        key = (solver.prob.ni, solver.prob.nj, solver.Nv, solver.precision)
        if key in self.cache:
            solver.set_tuning(**self.cache[key])
            return self.cache[key]
        G, H, W = solver.get_state()
        best, best_t = None, float("inf")
        # the micro sweeps' prefetch depth also decides how many velocity
        # tiles fit on the GPU at once (shared memory per block); the
        # macroscopic sweep keeps the deepest prefetch that fits
        own = {k: v for k, v in solver.tuning().items() if k != "graph"}  # the library's own choice first
        cands = [own] if own["sweep_vpt"] in self.candidates_vpt else []
        cands += [dict(sweep_tv=tv, sweep_vpt=vpt, sweep_stages=st, macro_stages=8)
                 for tv in self.candidates_tv for vpt in self.candidates_vpt for st in (2, 4, 8)]
        for cand in cands:
            try:
                solver.set_tuning(**cand)
            except B.IdgError:
                try:  # the macroscopic records may only fit a shallower prefetch
                    solver.set_tuning(**dict(cand, macro_stages=2))
                except B.IdgError:
                    continue
            solver.iterate_profiled()  # warm-up
            t = min(float(np.sum(solver.iterate_profiled())) for _ in range(self.repeats))
            if t < best_t:
                best, best_t = dict(solver.tuning()), t
        best.pop("graph", None)
        solver.set_tuning(**best)
        solver.set_state(G, H, W)  # timing iterations leave no trace
        self.cache[key] = best
        return best
