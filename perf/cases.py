"""The work this framework's users have it do, as cases that can be timed.

A case is a dict of plain values.  listed() gives the named cases, draw(rng) one more of the same
ranges, prepare(case, seed) what a program holds before the call (inputs on the GPU, plan,
workspace), run(state) one pass through the public entry points, work(case) what a pass cannot do
without, and exact(case, seed) the values of its floating-point outputs from torch in 64 bits.

Layouts are written as text: "aos", "soa", or groups of field numbers ("0,1|2|3"); field types as one
letter per field: f fp32, d fp64, i int32, h bf16.
"""
import collections
import math
import random

import torch

import paper_1407_4859_gb300 as P
from paper_1407_4859_gb300.autograd import DifferentiableProgram

SIZE = {"f": 4, "d": 8, "i": 4, "h": 2}
CODE = {"f": 0, "d": 1, "i": 2, "h": 3}
TORCH = {"f": torch.float32, "d": torch.float64, "i": torch.int32, "h": torch.int16}
DT = 2.0 ** -7

Section = collections.namedtuple("Section", "op args read write read_at_perm params table")


def section(op, args=(), read=(), write=(), at_perm=(), params=(), table=()):
    return Section(op, tuple(args), frozenset(read), frozenset(write), frozenset(at_perm), tuple(params), tuple(table))


# ------------------------------------------------------------------ the programs

STRESS = "ffffffffddddiiii"        # 80-byte records of three types
PARTICLES = "ffffffffiiid"         # 56-byte particles: position, velocity, mass, charge, id, cell, flags, energy
TINY = "ffffii"                    # 24-byte records
MEDICAL = "fffffffff"              # V1..V3, U1..U3, S, T, interpT
PARTICLE_GROUPS = "0,1,2,7|3,4,5|6|8|9|10|11"   # position and charge in one struct for the gather
MEDICAL_GROUPS = "0,1,2|3,4,5,7|6|8"


def tiny_sections():
    return [section("madd3", (0, 1, 2), (0, 1, 2), (2,)), section("xorshift", (4, 5), (3, 4), (5,)),
            section("add", (0, 3, 0), range(6), (0,))]


def stress_sections():
    """Eight sections touching about a third of the fields each, then one touching all of them."""
    rng, out = random.Random(1), []
    for _ in range(8):
        r = {f for f in range(16) if rng.random() < 0.3}
        w = {f for f in range(16) if rng.random() < 0.3} or {min(r) if r else 0}
        out.append(section("mix", (), r | w, w))
    return out + [section("mix", (), range(16), range(16))]


def particle_sections():
    drift = section("drift", range(6), range(6), range(3), params=(DT,))
    cell = section("bin", (0, 1, 2, 9), (0, 1, 2), (9,), params=(128.0,))
    ke = section("ke", (3, 4, 5, 6, 11), (3, 4, 5, 6), (11,))
    flags = section("flags", (10, 11), (10, 11), (10,), params=(1.5,))
    gather = section("gather", (3, 4, 5, 0, 1, 2, 7), (3, 4, 5), (3, 4, 5), (0, 1, 2, 7), params=(DT,))
    kick = section("kick", (3, 4, 5, 7), (3, 4, 5, 7), (3, 4, 5), params=(DT, 0.125, -0.0625, 0.03125))
    return [drift, cell, ke, flags, gather, kick, drift, cell, ke, flags]


def medical_sections():
    return [section("gather", (0, 1, 2, 3, 4, 5, 7), (0, 1, 2), (0, 1, 2), (3, 4, 5, 7), params=(DT,)),
            section("kick", (0, 1, 2, 6), (0, 1, 2, 6), (0, 1, 2), params=(DT, 0.25, -0.125, 0.0625)),
            section("drift", (3, 4, 5, 0, 1, 2), range(6), (3, 4, 5), params=(DT,)),
            section("axpb", (7, 8), (7,), (8,), params=(0.75, 0.125)),
            section("mul", (7, 8, 6), (7, 8), (6,)),
            section("madd3", (3, 0, 7), (0, 3, 7), (7,)),
            section("tanh", (6, 8), (6,), (8,))]


def kmeans_sections(d, k):
    rng = random.Random(6)
    cent = [rng.uniform(-1.0, 1.0) for _ in range(k * d)]
    return [section("assign", (d, k), range(d), (d,), table=cent), section("reduce", (d, k), range(d + 1))]


def chain_sections(fields, count):
    rng, out = random.Random(4), []
    for _ in range(count):
        u, x, y, z = rng.random(), rng.randrange(fields), rng.randrange(fields), rng.randrange(fields)
        if u < 0.4:
            out.append(section("axpb", (x, z), (x,), (z,), params=(rng.uniform(-1, 1), rng.uniform(-1, 1))))
        elif u < 0.7:
            out.append(section("mul", (x, y, z), (x, y), (z,)))
        else:
            out.append(section("tanh", (x, z), (x,), (z,)))
    return out


def program(case):
    """(field types, sections) of a program case."""
    return {"tiny": lambda: (TINY, tiny_sections()), "stress": lambda: (STRESS, stress_sections()),
            "particles": lambda: (PARTICLES, particle_sections()), "medical": lambda: (MEDICAL, medical_sections()),
            "kmeans": lambda: ("f" * case["features"] + "i", kmeans_sections(case["features"], case["clusters"])),
            }[case["program"]]()


# ------------------------------------------------------------------ cases

def listed():
    return [
        # the smallest whole program (the test suite's first configuration): remap and three sections, all latency
        dict(name="tiny_program", kind="program", program="tiny", n=65536, layout="soa", fused=False, specialised=False),
        # one small record array changed from structs to a gather-friendly layout: a single call's latency
        dict(name="remap_small", kind="remap", types=PARTICLES, src="aos", dst=PARTICLE_GROUPS, n=4099),
        # the large remap before a program's sections: 2^24 records of three types, structs to one array per field
        dict(name="remap_large", kind="remap", types=STRESS, src="aos", dst="soa", n=1 << 24),
        # the way back: grouped particles into structs, an odd record count
        dict(name="remap_back", kind="remap", types=PARTICLES, src=PARTICLE_GROUPS, dst="aos", n=9999991),
        # many uneven arrays of random record types (bf16 among them) through a prepared plan, as repeated conversions run
        dict(name="batched_launch", kind="batched", arrays=256, lo=1 << 10, hi=1 << 20, one_call=False),
        # a handful of smaller arrays converted once: planning is part of the call
        dict(name="batched_one_call", kind="batched", arrays=32, lo=1 << 8, hi=1 << 14, one_call=True),
        # the benchmark's program at its size, each section specialised at run time as its autotuner picks
        dict(name="stress_program", kind="program", program="stress", n=1 << 24, layout="soa", fused=False, specialised=True),
        # its nine sections combined into one pass by the library's own kernel, an odd record count
        dict(name="stress_fused", kind="program", program="stress", n=4194307, layout="soa", fused=True, specialised=False),
        # particles with a gather in a hybrid layout, library kernels
        dict(name="particles_program", kind="program", program="particles", n=8388593, layout=PARTICLE_GROUPS, fused=False,
             specialised=False),
        # K-Means step at the paper's size: nearest centroid, then per-cluster sums, in structs
        dict(name="kmeans_program", kind="program", program="kmeans", n=8388608, features=32, clusters=5, layout="aos",
             fused=False, specialised=False),
        # forward and backward of a 64-section differentiable chain through autograd
        dict(name="train_step", kind="train", n=1 << 24, fields=24, sections=64, layout="soa"),
        # the benchmark's program end to end from pinned host buffers, sliced over three streams
        dict(name="host_program", kind="program", program="stress", n=1 << 22, layout="soa", fused=False, specialised=False,
             slices=8),
    ]


def log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def partition(rng, fields, longest):
    order, out = list(range(fields)), []
    rng.shuffle(order)
    while order:
        k = rng.randint(1, longest)
        out.append(order[:k])
        order = order[k:]
    return "|".join(",".join(map(str, g)) for g in out)


def draw(rng):
    kind = rng.choice(["tiny", "remap", "remap", "batched", "one_call", "stress", "particles", "medical", "kmeans", "kmeans",
                       "train", "host"])
    if kind == "remap":
        types = "".join(rng.choice("fdih") for _ in range(rng.randint(4, 32)))
        sides = ["aos", rng.choice(["soa", partition(rng, len(types), 8)])]
        rng.shuffle(sides)
        n = log_int(rng, 1 << 10, (1 << 24) * 80 // max(80, sum(SIZE[t] for t in types) * 5 // 4))
        return dict(kind="remap", types=types, src=sides[0], dst=sides[1], n=n)
    if kind in ("batched", "one_call"):
        one = kind == "one_call"
        return dict(kind="batched", arrays=rng.randint(2, 32 if one else 256), lo=1 << 8, hi=log_int(rng, 1 << 10, 1 << (14 if one else 20)),
                    one_call=one)
    if kind == "train":
        layout = rng.choice(["soa", "soa", "aos"])
        return dict(kind="train", n=log_int(rng, 1 << 16, 1 << (24 if layout == "soa" else 20)), fields=24,
                    sections=rng.randint(8, 64), layout=layout)
    if kind == "kmeans":
        d = rng.randint(2, 32)
        return dict(kind="program", program="kmeans", n=log_int(rng, 1 << 12, 1 << 23), features=d, clusters=rng.randint(1, 8),
                    layout=rng.choice(["aos", "aos", "soa", partition(rng, d + 1, 8)]), fused=rng.random() < 0.25,
                    specialised=False)
    if kind == "tiny":
        return dict(kind="program", program="tiny", n=log_int(rng, 1 << 10, 1 << 17), layout=rng.choice(["soa", "aos"]),
                    fused=rng.random() < 0.3, specialised=False)
    if kind == "host":
        return dict(kind="program", program="stress", n=log_int(rng, 1 << 18, 1 << 22), layout="soa", fused=False,
                    specialised=False, slices=rng.choice([1, 4, 8]))
    if kind == "stress":
        return dict(kind="program", program="stress", n=log_int(rng, 1 << 16, 1 << 24),
                    layout=rng.choice(["soa", "0,1,2,3|4,5,6,7|8,9|10,11|12,13|14,15"]), fused=rng.random() < 0.5,
                    specialised=rng.random() < 0.5)
    groups = PARTICLE_GROUPS if kind == "particles" else MEDICAL_GROUPS
    return dict(kind="program", program=kind, n=log_int(rng, 1 << 14, 1 << 23), layout=rng.choice([groups, groups, "soa"]),
                fused=False, specialised=False)


# ------------------------------------------------------------------ inputs

def groups_of(text, fields):
    if text == "aos":
        return [list(range(fields))]
    if text == "soa":
        return [[f] for f in range(fields)]
    return [[int(f) for f in g.split(",")] for g in text.split("|")]


def struct_of(types, group):
    """(struct size, {field: byte offset}) of one group: C rules."""
    pos, align, off = 0, 1, {}
    for f in group:
        size = SIZE[types[f]]
        pos = (pos + size - 1) // size * size
        off[f] = pos
        pos += size
        align = max(align, size)
    return (pos + align - 1) // align * align, off


def field_views(types, groups, bufs):
    """One typed (strided) view per field, in field order."""
    out = [None] * len(types)
    for g, b in zip(groups, bufs):
        stride, off = struct_of(types, g)
        for f in g:
            size = SIZE[types[f]]
            out[f] = b.view(TORCH[types[f]]).view(-1, stride // size)[:, off[f] // size]
    return out


def pack(types, groups, n, values):
    """Group buffers (zero padding) holding the fields' values."""
    bufs = [torch.zeros(n * struct_of(types, g)[0], dtype=torch.uint8, device="cuda") for g in groups]
    for v, x in zip(field_views(types, groups, bufs), values):
        v.copy_(x)
    return bufs


def generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def raw_values(types, n, gen):
    out = []
    for t in types:
        v = torch.randint(-(1 << 15), 1 << 15, (n * SIZE[t] // 2,), dtype=torch.int16, device="cuda", generator=gen)
        out.append(v.view({4: torch.int32, 8: torch.int64, 2: torch.int16}[SIZE[t]]))
    return out


def program_values(case, types, gen):
    """Field values of a program's input records."""
    n = case["n"]

    def unit(dtype=torch.float32):
        return torch.rand(n, dtype=dtype, device="cuda", generator=gen)

    def normal():
        return torch.randn(n, device="cuda", generator=gen)

    def ints(hi=1 << 20):
        return torch.randint(0, hi, (n,), dtype=torch.int32, device="cuda", generator=gen)

    def zero(t):
        return torch.zeros(n, dtype=TORCH[t], device="cuda")

    name = case["program"]
    if name in ("tiny", "stress"):
        return [ints() if t == "i" else 2 * unit(TORCH[t]) - 1 for t in types]
    if name == "kmeans":
        return [2 * unit() - 1 for _ in range(case["features"])] + [zero("i")]
    if name == "medical":
        return [normal() for _ in range(3)] + [unit() for _ in range(3)] + [2 * unit() - 1 for _ in range(3)]
    return ([unit() for _ in range(3)] + [normal() for _ in range(3)] + [torch.exp(normal()), 2.0 * ints(2).float() - 1]
            + [torch.arange(n, dtype=torch.int32, device="cuda"), zero("i"), zero("i"), zero("d")])


def permutation(case, gen):
    if case["program"] not in ("particles", "medical"):
        return None
    return torch.randperm(case["n"], device="cuda", generator=gen).to(torch.int32)


def batched_arrays(case):
    """(types, target groups, n) of every array: 4..32 fields of random types, groups of 1..8 fields."""
    rng, out = random.Random(3), []
    for _ in range(case["arrays"]):
        types = "".join(rng.choice("fdih") for _ in range(rng.randint(4, 32)))
        out.append((types, partition(rng, len(types), 8), log_int(rng, case["lo"], case["hi"])))
    return out


def empty_groups(types, groups, n):
    return [torch.empty(n * struct_of(types, g)[0], dtype=torch.uint8, device="cuda") for g in groups]


def round256(x):
    return (x + 255) // 256 * 256


def prepare(case, seed):
    gen = generator(seed)
    return {"remap": prepare_remap, "batched": prepare_batched, "program": prepare_program,
            "train": prepare_train}[case["kind"]](case, gen)


def schema(types):
    return P.Schema([CODE[t] for t in types])


def prepare_remap(case, gen):
    types, n = case["types"], case["n"]
    src, dst = groups_of(case["src"], len(types)), groups_of(case["dst"], len(types))
    values = raw_values(types, n, gen)
    bufs = pack(types, src, n, [v.view(TORCH[t]) for v, t in zip(values, types)])
    return dict(kind="remap", schema=schema(types), n=n, src=P.Layout(src), src_bufs=bufs, dst=P.Layout(dst),
                dst_bufs=empty_groups(types, dst, n))


def prepare_batched(case, gen):
    plans = [(types, groups_of(target, len(types)), n) for types, target, n in batched_arrays(case)]
    # every destination group in one block of memory, as a program that owns all these arrays lays them out
    block = torch.zeros(sum(round256(n * struct_of(types, g)[0]) for types, dst, n in plans for g in dst), dtype=torch.uint8,
                        device="cuda")
    arrays, at = [], 0
    for types, dst, n in plans:
        dst_bufs = []
        for g in dst:
            size = n * struct_of(types, g)[0]
            dst_bufs.append(block[at:at + size])
            at += round256(size)
        stride = struct_of(types, list(range(len(types))))[0]
        src = torch.randint(0, 256, (n * stride,), dtype=torch.uint8, device="cuda", generator=gen)
        arrays.append(dict(schema=schema(types), n=n, src=P.Layout.aos(len(types)), src_bufs=[src], dst=P.Layout(dst),
                           dst_bufs=dst_bufs))
    state = dict(kind="one_call" if case["one_call"] else "batched", arrays=arrays, out=block)
    if case["one_call"]:
        state["workspace"] = torch.empty(P.adha_workspace_bytes(arrays), dtype=torch.uint8, device="cuda")
    else:
        state["plan"] = P.Batched(arrays)
        state["plan"].upload()
    return state


def prepare_program(case, gen):
    types, secs = program(case)
    n, F = case["n"], len(types)
    values = program_values(case, types, gen)
    perm = permutation(case, gen)
    bufs = pack(types, groups_of("aos", F), n, values)
    del values
    s, groups = schema(types), groups_of(case["layout"], F)
    cand = P.adha_layout_set_create(F, [P.Layout(groups)])
    sections = P.Sections(secs, perm=perm)
    state = dict(kind="program", schema=s, n=n, types=types, groups=groups, bufs=bufs, cand=cand, sections=sections,
                 aos=P.Layout.aos(F), fixed=[0] * len(secs), specialised=case["specialised"], key=None, out=None,
                 windows=[len(secs)] + [0] * (len(secs) - 1) if case["fused"] else None, plan=P._lib.adha_plan(),
                 opts=P.PlanOpts())
    if "slices" in case:
        k = case["slices"]
        state.update(kind="host", slices=k,
                     host_in=[b.cpu().pin_memory() for b in bufs],
                     host_out=[torch.empty(n * struct_of(types, g)[0], dtype=torch.uint8).pin_memory() for g in groups],
                     workspace=torch.empty(P.adha_program_host_workspace_bytes(s, n, state["aos"], cand, k),
                                           dtype=torch.uint8, device="cuda"))
        del state["bufs"]
        state["out"] = field_views(types, groups, state["host_out"])
    else:
        state["workspace"] = torch.empty(P.adha_program_workspace_bytes(s, n, state["aos"], cand), dtype=torch.uint8,
                                         device="cuda")
    return state


def chain_inputs(case, gen):
    return torch.randn((case["n"], case["fields"]), device="cuda", generator=gen)


def loss_weights(case):
    rng = random.Random(5)
    return [rng.uniform(-1.0, 1.0) for _ in range(case["fields"])]


def prepare_train(case, gen):
    F, n = case["fields"], case["n"]
    layout = P.Layout(groups_of(case["layout"], F))
    secs = chain_sections(F, case["sections"])
    c = loss_weights(case)
    seeds = [torch.tensor([c[f] for f in g], device="cuda").expand(n, len(g)).contiguous() for g in layout.groups]
    return dict(kind="train", x=chain_inputs(case, gen).requires_grad_(), seeds=seeds,
                program=DifferentiableProgram(schema("f" * F), n, P.Layout.aos(F), secs, [layout] * len(secs)))


# ------------------------------------------------------------------ one pass

def run(state):
    kind = state["kind"]
    if kind == "remap":
        P.adha_remap(state["schema"], state["n"], state["src"], state["src_bufs"], state["dst"], state["dst_bufs"])
        return state["dst_bufs"]
    if kind == "batched":
        state["plan"].launch()
        return state["out"]
    if kind == "one_call":
        P.adha_remap_batched(state["arrays"], state["workspace"])
        return state["out"]
    if kind == "train":
        x = state["x"]
        x.grad = None
        # the linear loss sum_f c_f sum_i x_f: its gradient with respect to the result is the constant c_f
        _, result = state["program"].forward([x])
        torch.autograd.backward(result, state["seeds"])
        return x.grad
    return run_program(state)


def run_program(state):
    if state["specialised"]:
        P.adha_tune_section_jit(2)
        P.adha_tune_fused_jit(2)
    try:
        if state["kind"] == "host":
            P.adha_run_program_host(state["schema"], state["n"], state["aos"], state["host_in"], state["sections"],
                                    state["cand"], state["host_out"], opts=state["opts"], workspace=state["workspace"],
                                    n_slices=state["slices"], fixed=state["fixed"], plan=state["plan"])
            return state["out"]
        plan = P.adha_run_program(state["schema"], state["n"], state["aos"], state["bufs"], state["sections"], state["cand"],
                                  opts=state["opts"], workspace=state["workspace"], fixed=state["fixed"],
                                  plan=state["plan"], windows=state["windows"])
    finally:
        if state["specialised"]:
            P.adha_tune_section_jit(0)
            P.adha_tune_fused_jit(0)
    # where the result lies (in the input buffers or the workspace): looked up again only when it moved
    key = plan.final_ptrs[:plan.final_n_groups]
    if key != state["key"]:
        bufs = []
        for ptr, g in zip(key, state["groups"]):
            owner = [b for b in state["bufs"] + [state["workspace"]] if b.data_ptr() <= ptr < b.data_ptr() + b.numel()][0]
            at = ptr - owner.data_ptr()
            bufs.append(owner[at:at + state["n"] * struct_of(state["types"], g)[0]])
        state["key"], state["out"] = key, field_views(state["types"], state["groups"], bufs)
        state["out"] += list(state["sections"].outputs.values())
    return state["out"]


# ------------------------------------------------------------------ work and exact values

OPS_PER_RECORD = dict(madd3=2, xorshift=2, add=1, drift=9, bin=15, ke=8, flags=3, gather=10, kick=7, axpb=2, mul=1, tanh=28)


def section_ops(types, s):
    if s.op == "mix":
        return len(s.read) + 3 + 2 * len(s.write)
    if s.op == "assign":
        return 3 * len(s.read) * s.args[1] + s.args[1]
    if s.op == "reduce":
        return 3 * len(s.read)
    return OPS_PER_RECORD[s.op]


def work(case):
    if case["kind"] == "remap":
        return dict(bytes=2 * case["n"] * sum(SIZE[t] for t in case["types"]), flops=0)
    if case["kind"] == "batched":
        return dict(bytes=sum(2 * n * sum(SIZE[t] for t in types) for types, _, n in batched_arrays(case)), flops=0)
    n = case["n"]
    if case["kind"] == "train":
        # the input records and their gradients; the program's state in between is the method's own
        flops = sum(3 * section_ops(None, s) for s in chain_sections(case["fields"], case["sections"]))
        return dict(bytes=2 * n * 4 * case["fields"], flops=n * flops)
    types, secs = program(case)
    data = sum(SIZE[t] for t in types)
    gathers = any(s.op == "gather" for s in secs)
    written = data
    if case["layout"] == "aos":   # the sections update the records where they are
        written = sum(SIZE[types[f]] for f in frozenset().union(*[s.write for s in secs]))
        data = sum(SIZE[types[f]] for f in frozenset().union(*[s.read | s.write for s in secs]))
        if case["program"] == "kmeans":   # the membership is not an input
            data -= 4
    return dict(bytes=n * (data + written + (4 if gathers else 0)), flops=n * sum(section_ops(types, s) for s in secs))


def exact(case, seed):
    gen = generator(seed)
    if case["kind"] == "train":
        return exact_train(case, gen)
    # remaps move bytes; the mix sections are defined over fp32 bit patterns, the K-Means sections give integers
    if case["kind"] != "program" or case["program"] in ("stress", "kmeans"):
        return None
    types, secs = program(case)
    x = [v.double() for v in program_values(case, types, gen)]
    perm = permutation(case, gen)
    for s in secs:
        exact_section(s, x, None if perm is None else perm.long())
    return [v if t in "fd" else None for v, t in zip(x, types)]


def exact_section(s, x, perm):
    a, p = s.args, [float(torch.tensor(v, dtype=torch.float32)) for v in s.params]
    if s.op == "madd3":
        x[a[2]] = x[a[0]] * x[a[1]] + x[a[2]]
    elif s.op == "add":
        x[a[2]] = x[a[0]] + x[a[1]]
    elif s.op == "drift":
        for k in range(3):
            q = x[a[k]] + p[0] * x[a[3 + k]]
            x[a[k]] = torch.where(q >= 1, q - 1, torch.where(q < 0, q + 1, q))
    elif s.op == "ke":
        x[a[4]] = 0.5 * x[a[3]] * (x[a[0]] ** 2 + x[a[1]] ** 2 + x[a[2]] ** 2)
    elif s.op == "gather":
        for k in range(3):
            x[a[k]] = x[a[k]] + p[0] * x[a[6]][perm] * (x[a[3 + k]][perm] - 0.5)
    elif s.op == "kick":
        for k in range(3):
            x[a[k]] = x[a[k]] + p[0] * x[a[3]] * p[1 + k]
    elif s.op == "axpb":
        x[a[1]] = p[0] * x[a[0]] + p[1]
    elif s.op == "mul":
        x[a[2]] = x[a[0]] * x[a[1]]
    elif s.op == "tanh":
        x[a[1]] = torch.tanh(x[a[0]])
    # xorshift, bin and flags write whole numbers only


def exact_train(case, gen):
    x0 = chain_inputs(case, gen)
    grad = torch.empty(x0.shape, dtype=torch.float64, device="cuda")
    step = 1 << 21   # by record range: the chain is per record
    c = [float(torch.tensor(v, dtype=torch.float32)) for v in loss_weights(case)]
    for i in range(0, case["n"], step):
        leaf = x0[i:i + step].double().requires_grad_()
        x = list(leaf.unbind(1))
        for s in chain_sections(case["fields"], case["sections"]):
            exact_section(s, x, None)
        sum(cf * xf.sum() for cf, xf in zip(c, x)).backward()
        grad[i:i + step] = leaf.grad
    return grad
