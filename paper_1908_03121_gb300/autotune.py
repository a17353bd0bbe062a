"""Autotuner for the same-level kernels' launch shapes.

Times whole solve steps (``Solver.step``: the passes overlapped on two streams,
so co-resident kernels share SMs as they will in the real step) on the
caller's tree for every candidate of
``fmm_tuning`` (sub-grids per pass of the monopole kernel, persistent CTAs per
SM, the dataflow downward pass or the level-by-level one, one or two multipole
target cells per thread in flight, the multipole work items the library picks
by the tree's size, whole or half sub-grids), each captured as a CUDA graph and
replayed, with CUDA events on the current stream; keeps the fastest and leaves
it set on the tree.  Each candidate is replayed ``reps`` times after one warm-up; the four fastest are
then timed again, round-robin, with about 100 ms of steps each, and the
median decides.  Results are cached per tree size and precision for the
process.
"""

import itertools

import numpy as np

from . import fmm as B

MONO_SUBGRIDS = (1, 2, 4)
CTAS_PER_SM = (0, 1, 2)
DATAFLOW = (0, 1)
MP_ITEMS = (0, 1, 2)      # 0: by the tree's size
_CACHE = {}


def _key(solver):
    s = solver.tree.sizes
    return (s["n_nodes"], s["n_leaf"], s["n_refined"], s["precision"],
            int(solver.tree.stats["stencil_union"]), getattr(solver, "order", 3))


def candidates(precision, order, n_multipole, sms):
    """The tunings to time: every launch shape once.  ``n_multipole``: refined
    sub-grids below the roots (the multipole launch's), ``sms``: the GPU's SMs.
    What a precision's kernels do not read stays at its default."""
    mixed = precision == B.FMM_MIXED
    if precision == B.FMM_FP64:
        items = (0,)         # long steps: automatic
    elif mixed:
        # by size has shapes of its own up to one sub-grid an SM, above it is one of the others
        items = MP_ITEMS if n_multipole <= sms else MP_ITEMS[1:]
    else:
        # sixteenths, whatever is asked for, where quarters do not fill the SMs
        items = MP_ITEMS[1:] if 4 * n_multipole >= sms else (0,)
    shapes = [(0, it) for it in items] + ([(1, 0)] if mixed and order == 3 else [])
    return [dict(mono_subgrids=nb, ctas_per_sm=cap, dataflow=df, mp_pair_targets=pt, mp_items=it)
            for nb, cap, df, (pt, it) in itertools.product(MONO_SUBGRIDS if mixed else (0,), CTAS_PER_SM,
                                                           DATAFLOW, shapes)]


def tune(solver, reps=5, verbose=False, flush=None, graph=True):
    """Pick and set the fastest tuning for ``solver`` (an ``fmm.Solver``).
    ``flush``, if given, is called before every timed step (the benchmark's
    L2 flush, so that candidates are compared as the benchmark times them).
    ``graph``: time replays of the step captured as a CUDA graph under each
    candidate (as the benchmark and ``Solver.replay`` run it), else eager
    steps.  Leaves ``solver.graph`` unset: capture again after tuning."""
    import torch
    key = _key(solver)
    if key in _CACHE:
        B.fmm_set_tuning(solver.tree, **_CACHE[key][0])
        return _CACHE[key]
    stream = torch.cuda.current_stream()

    def runner(cand):
        # the step as the caller will run it: one CUDA graph captured under
        # this tuning (launch shapes are fixed at capture), replayed; eager
        # steps would add launch costs that a replay does not pay, which
        # favours the shapes with fewer launches
        B.fmm_set_tuning(solver.tree, **cand)
        g = solver.capture() if graph else None
        run = g.replay if g is not None else solver.step
        run()
        return g, run

    def timed(run):
        if flush is not None:
            flush()
        a = torch.cuda.Event(enable_timing=True)
        b = torch.cuda.Event(enable_timing=True)
        a.record(stream)
        run()
        b.record(stream)
        b.synchronize()
        return a.elapsed_time(b)

    results = []
    sms = torch.cuda.get_device_properties(stream.device).multi_processor_count
    for cand in candidates(solver.tree.sizes["precision"], getattr(solver, "order", 3),
                           solver.tree.stats["work_items"][0], sms):
        g, run = runner(cand)
        times = [timed(run) for _ in range(reps)]
        del g
        results.append((float(np.median(times)), cand))
        if verbose:
            print(f"  {cand}: {np.median(times):.3f} ms")
    results.sort(key=lambda r: r[0])
    # The four fastest again, round-robin (so that clock or cache drift
    # falls on all of them alike), with about 100 ms of steps each: the first
    # pass's few steps cannot tell shapes within a percent apart.
    top = [c for _, c in results[:4]]
    runs = [runner(c) for c in top]
    more = max(reps, min(200, int(100.0 / max(results[0][0], 1e-3))))
    again = [[] for _ in top]
    for _ in range(more):
        for i, (_, run) in enumerate(runs):
            again[i].append(timed(run))
    del runs
    final = sorted(((float(np.median(t)), c) for t, c in zip(again, top)), key=lambda r: r[0])
    if verbose:
        for ms, c in final:
            print(f"  again {c}: {ms:.3f} ms")
    best = final[0][1]
    B.fmm_set_tuning(solver.tree, **best)
    solver.graph = None
    _CACHE[key] = (best, final + results[len(top):])
    return _CACHE[key]
