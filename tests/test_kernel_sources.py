"""Rules of the CUDA sources that no run can show, because the compiler may happen to hide their violation: checked on the text."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_00404_b200", "csrc")


def _sources():
    """(file, line number, code) of every line, comments removed."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as f:
            for i, line in enumerate(f, 1):
                out.append((os.path.basename(path), i, line.split("//")[0]))
    assert len(out) > 1000
    return out


def test_no_exchange_takes_its_mask_from_the_lanes_that_happen_to_be_active():
    """__activemask() does not bring a warp together: a lane whose partner has not arrived yet would exchange with nothing."""
    assert [(f, i) for f, i, code in _sources() if "__activemask" in code] == []


def test_nothing_is_summed_in_the_order_of_arrival():
    """The library repeats itself bit for bit, so its atomic additions are on integers."""
    adds = [(f, i, code.strip()) for f, i, code in _sources() if re.search(r"\batomicAdd\b|\bred\.[a-z.]*add", code)]
    assert [a for a in adds if "eig_norm2_units(" not in a[2]] == []
    decl = [code for _, _, code in _sources() if re.search(r"\bnorm2\[ER_STEPS\]", code)]
    assert len(decl) == 1 and "unsigned long long" in decl[0]


def test_tensor_copies_of_codes_are_checked_in_the_debug_build():
    """A tensor copy that leaves its matrix is clipped by the hardware, so nothing else would show it: both of its ranges stand behind
    the debug build's check."""
    with open(os.path.join(CSRC, "residual_tc.cu")) as f:
        code = re.sub(r"//[^\n]*", "", f.read())
    copies = [m.start() for m in re.finditer(r"\btma_store_2d\(", code)]
    assert len(copies) == 2
    for at in copies:
        statement = code[code.rfind(";", 0, at):at]
        assert re.findall(r"METIS_DBG_GUARD\([^,]*, [^,]*, (\d+), ", statement) == ["16", "32"], statement


def _constants(text, known):
    """Values of the `constexpr int` names that `text` declares, `known` given (conditional expressions become Python's)."""
    out = dict(known)
    for statement in re.findall(r"constexpr int ([^;(]*(?:\([^;]*\))?[^;]*);", text):
        for name, expr in re.findall(r"(\w+) = ([^,]+)", statement):
            expr = re.sub(r"\w+::", "", expr.replace("&&", " and ").replace("||", " or ")).strip()
            expr = re.sub(r"^(.+?) \? (.+) : (.+)$", r"(\2) if (\1) else (\3)", expr.replace("(TAIL ? WT_TAIL : 0)", "(WT_TAIL if TAIL else 0)"))
            try:
                out[name] = int(eval(expr.replace("/", "//"), {}, out))
            except (NameError, SyntaxError):
                pass                                       # made of something else than integers known here
    return out


def test_arrays_of_the_reduction_hold_an_entry_for_every_row_of_an_instance():
    """tridiag_chol_kernel works on WT_WARPS * R rows, whether or not they belong to the matrix, and indexes two shared arrays with
    them.  Out of range, an access falls into a neighbouring array, which no run shows."""
    with open(os.path.join(CSRC, "bigrank.cuh")) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    with open(os.path.join(CSRC, "split.cu")) as f:
        launches = re.sub(r"//[^\n]*", "", f.read())
    kernel = text[text.index("tridiag_chol_kernel(const"):]
    kernel = kernel[:kernel.index("\n}\n")]
    shape = re.search(r"struct WtShape \{(.*?)\n\};", text, re.S)
    for name in ("ys", "pq"):
        assert re.findall(r"\b%s\[([^\]]*WT_WARPS[^\]]*)\]" % name, kernel)
    instances = re.findall(r"launch_tridiag<(?:[^<>]*, )??(\d+), (\d+), (true|false)>\(s,", launches)
    assert len(instances) == 4
    for r, c, tail in instances:
        known = _constants(text[text.index("constexpr int WT_WARPS"):text.index("struct WtShape" if shape else "template <int R, int C, bool TAIL>")],
                           {"R": int(r), "C": int(c), "TAIL": tail == "true"})
        known = _constants((shape.group(1) if shape else "") + kernel, known)
        rows = 15 * int(r)                                 # warp + WT_WARPS * a, a < R
        assert known["WT_WARPS"] == 15
        for name in ("ys", "pq"):
            extent = re.search(r"__shared__[^;]*\b%s\[([^\]]+)\]" % name, kernel).group(1)
            assert eval(re.sub(r"\w+::", "", extent), {}, known) >= rows, (name, r, c, tail)
        if tail == "true":
            assert rows <= known["WT_MAX"] + known["WT_WARPS"]                 # rows of `tail`


def test_shared_arrays_accessed_in_vectors_are_declared_aligned():
    """A 16- (8-) byte access to a shared array of smaller elements needs the declaration to say so: without it the array lies where
    the others leave room."""
    size = {"double2": 16, "float4": 16, "uint4": 16, "int4": 16, "float2": 8, "uint2": 8, "int2": 8}
    wanted, found = 0, []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for kernel in re.split(r"\b__global__\b", text)[1:]:
            align = {"smem_raw": 1024} if "(raw + 1023u) & ~1023u" in kernel else {}   # rounded up by the kernel itself
            for decl in re.findall(r"__shared__[^;]*;", kernel):
                a = re.search(r"__align__\((\d+)\)", decl)
                base = 8 if re.search(r"\b(double|float2|uint2|uint64_t)\b", decl) else (16 if re.search(r"\b(double2|float4|uint4)\b", decl) else 4)
                for name in re.findall(r"\b(\w+)\[", decl):
                    align.setdefault(name, max(base, int(a.group(1)) if a else 0))
            source = dict(re.findall(r"\*\s*(?:__restrict__ )?(\w+) = (?:reinterpret_cast<[^;=]*>\()?&?(\w+)\b(?![(])", kernel))
            for type_, name in re.findall(r"reinterpret_cast<(?:const )?(\w+)\s*\*>\(\s*&?(\w+)", kernel):
                for _ in range(4):
                    if name in align or name not in source:
                        break
                    name = source[name]
                if type_ in size and name in align:
                    wanted += 1
                    if align[name] < size[type_]:
                        found.append((os.path.basename(path), type_, name))
    assert wanted >= 10
    assert found == []


def _body(text, head):
    """What stands between the braces behind `head`."""
    at = text.index("{", text.index(head) + len(head) - 1)
    depth, end = 0, at
    while True:
        depth += {"{": 1, "}": -1}.get(text[end], 0)
        end += 1
        if depth == 0:
            return text[at + 1:end - 1]


def _shared_events(body, pairs, step):
    """The barrier calls and the accesses to shared vectors of one step of a loop, in order: ("arrive" | "await", barrier) and
    ("read" | "write", vector, half).  pairs: the vectors with two halves; a pointer that is set to one of them stands for it."""
    def value(expr):
        return eval(expr, {}, {"j": step})

    alias, events = {}, []
    name = r"ys|us|ps|qs|rs|V"
    for m in re.finditer(r"\b(?P<decl>\w+) = (?P<of>rs|ps)\[(?P<dh>[^\]]*)\](?: \+ \w+)?[,;]|\b(?P<sync>arrive|await)\((?P<bar>\w+)\)"
                         r"|reinterpret_cast<(?P<const>const )?double2\*>\((?P<cast>%s)(?:\[(?P<ch>[^\]]*)\])? \+ [^)]*\)"
                         r"|\b(?P<vec>%s|rj|out)\[(?P<idx>[^\]]*)\](?:\[[^\]]*\])?(?P<set> = )?" % (name, name), body):
        if m["decl"]:
            alias[m["decl"]] = (m["of"], value(m["dh"]))
        elif m["sync"]:
            events.append((m["sync"], m["bar"]))
        elif m["cast"]:
            events.append(("read" if m["const"] else "write", m["cast"], value(m["ch"]) if m["cast"] in pairs else 0))
        else:
            vec, half = alias.get(m["vec"], (m["vec"], None))
            if half is None:
                half = value(m["idx"]) if vec in pairs else (value(m["idx"].split(" * P")[0]) if vec == "V" else 0)
            events.append(("write" if m["set"] else "read", vec, half))
    return events


def test_vectors_of_the_one_cta_reduction_change_hands_behind_a_barrier():
    """The rows' warps and the scalars' warp of eig_kernel run a step or so apart, joined by one-sided barriers: of two accesses to a
    shared vector from either side, one of which writes, one has to happen before the other by the barriers alone, whatever the warps' pace."""
    with open(os.path.join(CSRC, "small_eig.cuh")) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    kernel = text[text.index("eig_kernel(const double"):]
    pairs = set(re.findall(r"\b(\w+)\[2\]\[N8\]", re.search(r"__shared__[^;]*\bps\[[^;]*;", kernel).group(0)))
    loops = {"rows": _body(kernel, "for (int j = from; j < to; ++j) {"), "scalars": _body(kernel, "for (int j = 0; j + 2 < n; ++j) {")}
    # every event's position in its own side's order, and what of the other side has happened before it
    order, signals, steps = {}, {}, 6
    for side, body in loops.items():
        order[side] = [e for step in range(steps) for e in _shared_events(body, pairs, step)]
        seen = {}
        for at, e in enumerate(order[side]):
            if e[0] == "arrive":
                seen[e[1]] = seen.get(e[1], 0) + 1
                signals[side, e[1], seen[e[1]]] = at
    other = {"rows": "scalars", "scalars": "rows"}
    before = {}
    for side in order:                                     # before[side][at]: events of the other side up to here have happened
        seen, known, before[side] = {}, -1, []
        for e in order[side]:
            if e[0] == "await":
                seen[e[1]] = seen.get(e[1], 0) + 1
                known = max(known, signals[other[side], e[1], seen[e[1]]])
            before[side].append(known)
    found, shared = [], set()
    for a, x in enumerate(order["rows"]):
        for b, y in enumerate(order["scalars"]):
            if x[0] in ("read", "write") and x[1:] == y[1:] and "write" in (x[0], y[0]) and y[0] in ("read", "write"):
                shared.add(x[1])
                if before["rows"][a] < b and before["scalars"][b] < a:
                    found.append((x, a, y, b))
    assert shared == {"ys", "us", "ps", "qs", "rs", "V"}
    assert found == []
