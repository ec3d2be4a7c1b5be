"""Differentiation through layout changes and chains of fp32 sections.

State in a layout is a list of float32 tensors, one (n, k) tensor per group of k fields (all fields
fp32, so a group's struct is k contiguous floats).  Three autograd Functions:

* RemapFn: moves the groups that change from one layout to another with the remap kernel; its
  backward is the inverse remap of the incoming gradients (the same byte permutation, reversed).
  Groups the two layouts share are not inputs or outputs of the Function: the same tensor carries
  the data and its gradient straight through.
* SegmentFn: runs a run of axpb / mul / tanh sections in place in one layout, as chain runs
  (adha_chain_forward) that save what the written fields held before the run; its backward
  (adha_chain_backward) puts that back, runs the sections again on chip and walks them in reverse,
  propagating the adjoints.  A few sections on wide structs run one by one instead, each saving the
  value it overwrites, and its adjoint kernel (adha_section_backward) restores it.  (A schema with other
  types than fp32 runs forward that way too; there is no backward for it.)
* CopyFn: a copy of the state by the remap kernel, where the first section keeps the input layout.

DifferentiableProgram strings them together for a whole program under a layout plan.  Every
forward and backward step runs in the library's kernels; PyTorch only allocates and orders them.
Memory: the forward keeps one saved field (n floats) per written field of each chain run, or per section run
on its own, and every layout's moved groups;
the backward hands the program's state back to what it was before each segment, in place, so the
forward outputs hold the input-side values once backward() has run (copy them first if needed).
"""
import torch

from ._lib import adha_section
from .api import (adha_chain_backward, adha_chain_forward, adha_chain_plan, adha_remap, adha_run_section,
                  adha_section_backward, c_section)


def _copy(schema, n, layout, groups):
    """Fresh copies of a layout's group tensors, moved by the library's remap kernel (identical
    groups at different addresses are copied, not aliased)."""
    out = [torch.empty_like(g) for g in groups]
    adha_remap(schema, n, layout, list(groups), layout, out)
    return out


class CopyFn(torch.autograd.Function):
    """A copy of the state (sections then update the copy in place and leave the inputs intact);
    its backward passes the gradients through."""

    @staticmethod
    def forward(ctx, meta, *groups):
        schema, n, layout = meta
        return tuple(_copy(schema, n, layout, groups))

    @staticmethod
    def backward(ctx, *grads):
        return (None,) + grads


def _alias_map(src, dst):
    """dst group index -> src group index for groups identical in both layouts."""
    out = {}
    for d, g in enumerate(dst.groups):
        for s, h in enumerate(src.groups):
            if g == h:
                out[d] = s
    return out


class RemapFn(torch.autograd.Function):
    @staticmethod
    def forward(ctx, meta, *moved_src):
        schema, n, src, dst, src_all = meta
        alias = _alias_map(src, dst)
        moved_s = [s for s in range(len(src.groups)) if s not in alias.values()]
        src_ptrs = list(src_all)
        for k, s in enumerate(moved_s):
            src_ptrs[s] = moved_src[k]
        out = {}
        dst_ptrs = []
        for d, g in enumerate(dst.groups):
            if d in alias:
                dst_ptrs.append(src_ptrs[alias[d]])
            else:
                out[d] = torch.empty((n, len(g)), dtype=torch.float32, device="cuda")
                dst_ptrs.append(out[d])
        adha_remap(schema, n, src, src_ptrs, dst, dst_ptrs)
        ctx.meta = (schema, n, src, dst, alias, moved_s)
        return tuple(out[d] for d in sorted(out))

    @staticmethod
    def backward(ctx, *grads):
        schema, n, src, dst, alias, moved_s = ctx.meta
        moved_d = [d for d in range(len(dst.groups)) if d not in alias]
        gd = {}
        for k, d in enumerate(moved_d):
            g = grads[k]
            gd[d] = g.contiguous() if g is not None else torch.zeros((n, len(dst.groups[d])), dtype=torch.float32,
                                                                       device="cuda")
        gs = {s: torch.empty((n, len(src.groups[s])), dtype=torch.float32, device="cuda") for s in moved_s}
        # shared groups: one placeholder buffer on both sides, so the kernel leaves them alone
        placeholder = torch.empty(16, dtype=torch.uint8, device="cuda")
        d_ptrs = [gd[d] if d in gd else placeholder for d in range(len(dst.groups))]
        s_ptrs = []
        for s in range(len(src.groups)):
            if s in gs:
                s_ptrs.append(gs[s])
            else:
                d = [dd for dd, ss in alias.items() if ss == s][0]
                s_ptrs.append(d_ptrs[d])
        adha_remap(schema, n, dst, d_ptrs, src, s_ptrs)      # inverse remap of the gradients
        return (None,) + tuple(gs[s] for s in moved_s)


def _faster_one_by_one(n, layout, sections):
    """Whether a short segment on structs runs section by section: a chain run moves whole structs, a record
    per lane, however few of their fields it touches.  Modelled ns per record, from runs of 2^22 records: a
    chain run 0.0018 per byte of the structs it touches (0.0024 from 128 bytes on, 0.0037 where the size is
    no multiple of 16) and a copy of the other gradients; sections 0.022 per operand in a struct, 0.0005 per
    byte of the structs they read, and a copy of all gradients; and 0.03 ms of the host for a section's
    launches.  Forward + backward, chain run / one by one: 64 fields in a struct, 1 section 2886 / 1342 us, 2
    2882 / 2104, 3 2879 / 2783; 63 fields 1 section 4235 / 1294, 4 4280 / 3020; 24 fields 1 section 763 / 582."""
    copied = 8 * 1.55e-4   # a gradient's bytes, read and written, at the copy rate
    structs = [g for g in layout.groups if len(g) > 1]
    cost = [4 * len(g) * (0.0037 if len(g) % 4 else 0.0018 if len(g) < 32 else 0.0024) for g in structs]
    single = copied * sum(map(len, layout.groups))
    launches = 3e4 * (2 + len(sections))
    if n * (sum(cost) - single - 0.022 * len(sections)) <= launches:   # at most this, without a look at the operands
        return False
    at = {f: k for k, g in enumerate(structs) for f in g}
    run = set()
    for s in sections:
        operands = [at[f] for f in s.args if f in at]
        run.update(operands)
        single += 0.022 * len(operands) + 0.0005 * sum(4 * len(structs[k]) for k in set(operands))
    whole = sum(cost[k] if k in run else copied * len(structs[k]) for k in range(len(structs)))
    return n * (whole - single) > launches


class SegmentFn(torch.autograd.Function):
    @staticmethod
    def forward(ctx, meta, *groups):
        schema, n, layout, sections = meta
        runs = []
        k = 0
        # other types than fp32 (forward only): chain runs do not take them
        ctx.one_by_one = any(schema.dtypes) or _faster_one_by_one(n, layout, sections)
        if ctx.one_by_one:
            for s in sections:
                cs = c_section(s)
                save = torch.empty(n, dtype=torch.float32, device="cuda")
                adha_run_section(schema, n, layout, groups, cs, save=save)
                runs.append((cs, save))
            k = len(sections)
        while k < len(sections):
            secs = (adha_section * (len(sections) - k))(*[c_section(s) for s in sections[k:]])
            m, need = adha_chain_plan(schema, n, secs)
            if m < len(secs):
                secs = (adha_section * m)(*secs[:m])
            saved = torch.empty(need // 4, dtype=torch.float32, device="cuda")
            adha_chain_forward(schema, n, layout, groups, secs, saved)
            runs.append((secs, saved))
            k += m
        ctx.meta = (schema, n, layout)
        ctx.state = groups          # updated in place; the backward restores it run by run
        ctx.runs = runs
        ctx.mark_dirty(*groups)
        return groups

    @staticmethod
    def backward(ctx, *grads):
        schema, n, layout = ctx.meta
        g = [x.contiguous() if x is not None else torch.zeros((n, len(layout.groups[k])), dtype=torch.float32,
                                                              device="cuda")
             for k, x in enumerate(grads)]
        # the incoming gradients stay as they are: the last run's pass writes buffers of its own (the adjoint
        # kernel works in place, on copies), which the earlier ones then update in place
        if ctx.one_by_one or not ctx.runs:
            out = _copy(schema, n, layout, g)
            for cs, save in reversed(ctx.runs):
                adha_section_backward(schema, n, layout, ctx.state, out, cs, save)
        else:
            out = [torch.empty_like(x) for x in g]
            for secs, saved in reversed(ctx.runs):
                adha_chain_backward(schema, n, layout, ctx.state, g, out, secs, saved)
                g = out
        # the state tensors' grad_fn refers to ctx: drop them here, or the step's memory waits for
        # Python's cycle collector
        ctx.runs = None
        ctx.state = None
        return (None,) + tuple(out)


class DifferentiableProgram:
    """A chain of axpb / mul / tanh sections under a layout plan (one Layout per section)."""

    def __init__(self, schema, n, in_layout, sections, plan_layouts):
        for s in sections:
            if s.op not in ("axpb", "mul", "tanh"):
                raise ValueError("differentiable programs take axpb, mul and tanh sections (got %s)" % s.op)
        self.schema, self.n, self.in_layout = schema, n, in_layout
        self.sections = list(sections)
        self.plan = list(plan_layouts)

    def _remap(self, state, src, dst):
        alias = _alias_map(src, dst)
        moved_s = [s for s in range(len(src.groups)) if s not in alias.values()]
        outs = RemapFn.apply((self.schema, self.n, src, dst, list(state)), *[state[s] for s in moved_s])
        it = iter(outs)
        return [state[alias[d]] if d in alias else next(it) for d in range(len(dst.groups))]

    def forward(self, in_groups):
        """in_groups: (n, k) float32 tensors of the input layout.  Returns (final layout, groups)."""
        cur = self.in_layout
        state = list(in_groups)
        first = True
        k = 0
        while k < len(self.sections):
            lay = self.plan[k]
            j = k
            while j < len(self.sections) and self.plan[j] == lay:
                j += 1
            if lay != cur:
                state = self._remap(state, cur, lay)
                cur = lay
            elif first:
                state = list(CopyFn.apply((self.schema, self.n, cur), *state))   # leave the inputs intact
            first = False
            state = list(SegmentFn.apply((self.schema, self.n, cur, self.sections[k:j]), *state))
            k = j
        return cur, state
