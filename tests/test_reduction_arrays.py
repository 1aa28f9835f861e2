"""The reduction arrays of the fused kernel's shared memory (ClusterShared::red_*),
checked on the source: along every path through one CTA's work on its
clusters, a __syncthreads lies between two uses of an array whenever one of
them writes it.  A use without one is a race that a run hardly ever shows:
warps would have to drift apart by a whole pass over the points.

The walk expands the calls between the kernel's own functions and lambdas,
takes both sides of every branch and every loop twice.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2012_12618_gb300", "csrc")
TOKEN = re.compile(r"[A-Za-z_]\w*|\d[\w.]*|==|!=|<=|>=|&&|\|\||\+\+|--|[-+*/|&^]=|::|->|\S")
BARRIERS = ("__syncthreads", "__syncthreads_or")
CLOSE = {"(": ")", "[": "]", "{": "}"}


def tokens(text):
    text = re.sub(r"//[^\n]*|/\*.*?\*/", " ", text, flags=re.S)
    return TOKEN.findall("\n".join(l for l in text.splitlines() if not l.lstrip().startswith("#")))


def match(t, i):
    """Index of the bracket that closes t[i]."""
    depth = 0
    for k in range(i, len(t)):
        depth += t[k] in CLOSE
        depth -= t[k] in CLOSE.values()
        if depth == 0:
            return k
    raise AssertionError("unbalanced")


def functions(t):
    """name -> (parameter names, body tokens) of every function with a body."""
    out = {}
    for i in range(1, len(t) - 1):
        if t[i] != "(" or not re.match(r"[A-Za-z_]", t[i - 1]) or t[i - 1] in ("if", "for", "while", "switch"):
            continue
        end = match(t, i)
        if end + 1 < len(t) and t[end + 1] == "{" and re.match(r"[A-Za-z_>*&]", t[i - 2]):
            out[t[i - 1]] = (split_names(t[i + 1:end]), t[end + 2:match(t, end + 1)])
    return out


def split_args(t):
    args, depth = [[]], 0
    for x in t:
        depth += x in CLOSE
        depth -= x in CLOSE.values()
        if x == "," and depth == 0:
            args.append([])
        else:
            args[-1].append(x)
    return args


def split_names(t):
    names = []
    for a in split_args(t):
        a = a[:a.index("[")] if "[" in a else a  # array parameters
        names.append(a[-1] if a else "")
    return names


class Walk:
    """State: per array, the uses ("r", "w") since the last barrier."""

    def __init__(self, text):
        self.fns = functions(tokens(text))
        self.races = set()

    def use(self, state, array, kind, where):
        was = state.get(array, frozenset())
        if (kind == "w" and "r" in was) or (kind == "r" and "w" in was):
            self.races.add((where, array))
        state[array] = was | {kind}

    @staticmethod
    def join(*states):
        out = {}
        for s in states:
            for k, v in s.items():
                out[k] = out.get(k, frozenset()) | v
        return out

    # -- statements: returns the state after them; left: states of paths that left early
    def block(self, t, env, state, where, left):
        i = 0
        while i < len(t):
            i, state = self.statement(t, i, env, state, where, left)
        return state

    def statement(self, t, i, env, state, where, left):
        if t[i] == "{":
            end = match(t, i)
            return end + 1, self.block(t[i + 1:end], dict(env), state, where, left)
        if t[i] in ("if", "for", "while"):
            kw, j = t[i], i + 1
            j += t[j] == "constexpr"
            end = match(t, j)
            state = self.expr(t[j + 1:end], env, dict(state), where)
            if kw == "if":
                k, then = self.statement(t, end + 1, env, dict(state), where, left)
                if k < len(t) and t[k] == "else":
                    k, other = self.statement(t, k + 1, env, dict(state), where, left)
                    return k, self.join(then, other)
                return k, self.join(state, then)
            out = state
            for _ in range(2):
                inner = []
                k, state = self.statement(t, end + 1, env, dict(state), where, inner)
                state = self.join(state, *[s[1] for s in inner if s[0] == "continue"])
                state = self.expr(t[j + 1:end], env, state, where)
                left += [s for s in inner if s[0] == "return"]
                out = self.join(out, state, *[s[1] for s in inner if s[0] == "break"])
            return k, out
        end = i
        while end < len(t) and t[end] != ";":
            end = match(t, end) + 1 if t[end] in CLOSE else end + 1
        stmt = t[i:end]
        lam = stmt[:1] == ["auto"] and "=" in stmt and stmt[stmt.index("=") + 1:stmt.index("=") + 2] == ["["]
        if lam:
            p = stmt.index("(")
            b = stmt.index("{", match(stmt, p))
            rest = stmt[match(stmt, b) + 1:]
            if not rest:  # a named lambda: walked where it is called
                env[stmt[1]] = (split_names(stmt[p + 1:match(stmt, p)]), stmt[b + 1:match(stmt, b)], env)
                return end + 1, state
        state = self.expr(stmt, env, dict(state), where)
        if stmt and stmt[0] in ("return", "break", "continue"):
            left.append((stmt[0], state))
            state = {}
        return end + 1, state

    def array(self, t, i, env):
        """Array named at t[i] (cs.red_x or a parameter bound to one), and where its name ends."""
        if t[i] == "cs" and t[i + 1:i + 2] == ["."] and i + 2 < len(t) and t[i + 2].startswith("red_"):
            return t[i + 2], i + 3
        if isinstance(env.get(t[i]), str) and t[i - 1:i] != ["."]:
            return env[t[i]], i + 1
        return None, i

    def expr(self, t, env, state, where):
        i, writes = 0, []
        while i < len(t):
            if t[i] in BARRIERS:
                state = {}
            name, j = self.array(t, i, env) if t[i] == "cs" or t[i] in env else (None, i)
            if name:
                indexed = False
                while j < len(t) and t[j] == "[":
                    state = self.expr(t[j + 1:match(t, j)], env, state, where)
                    j = match(t, j) + 1
                    indexed = True
                if indexed and t[j:j + 1] == ["="]:
                    writes.append(name)
                else:  # read, or handed whole to a function that reads it
                    self.use(state, name, "r", where)
                i = j
                continue
            fn = env.get(t[i]) if isinstance(env.get(t[i]), tuple) else self.fns.get(t[i])
            if fn and t[i - 1:i] not in (["."], ["->"]):
                p = i + 1
                if t[p:p + 1] == ["<"]:  # template arguments
                    while p < len(t) and t[p] != "(":
                        p += 1
                        if t[p - 1] == "decltype":
                            p = match(t, p) + 1
                if t[p:p + 1] == ["("]:
                    end = match(t, p)
                    state = self.call(t[i], fn, split_args(t[p + 1:end]), env, state, where)
                    i = end + 1
                    continue
            i += 1
        for name in writes:
            self.use(state, name, "w", where)
        return state

    def call(self, fname, fn, args, env, state, where):
        params, body = fn[0], fn[1]
        new = dict(fn[2]) if len(fn) > 2 else {}
        for p, a in zip(params, args):
            new.pop(p, None)
            name, end = self.array(a, 0, env) if a else (None, 0)
            if name and end == len(a):
                new[p] = name
            else:
                state = self.expr(a, env, state, where)
        left = []
        after = self.block(body, new, state, where + "/" + fname, left)
        return self.join(after, *[s[1] for s in left])


def races(text):
    w = Walk(text)
    params, body = w.fns["process_cluster"]
    for needed in ("staged_pass", "prune_list", "block_best", "mask_and_sums", "block_median", "local_opt_rounds"):
        assert needed in w.fns, needed
    # one cluster: the kernel's loop over clusters has barriers between them
    w.block(body, {}, {}, "process_cluster", [])
    return sorted(w.races)


def source():
    with open(os.path.join(CSRC, "rvh_fused.cu")) as f:
        return f.read()


def test_every_reduction_array_has_its_barrier():
    assert races(source()) == []


PLANTED = {
    # a barrier less, or an array that may still be read
    "prune_list": ("    out += tot;\n    __syncthreads();\n", "    out += tot;\n"),
    "mask": ("    cs.red_c[warp] = nch;\n  }\n  __syncthreads();\n", "    cs.red_c[warp] = nch;\n  }\n"),
    "staged": ("cs.red_c[warp] = (int)cnt;", "cs.red_i[warp] = (int)cnt;"),
}


@pytest.mark.parametrize("name", list(PLANTED))
def test_a_planted_fault_is_found(name):
    text = source()
    old, new = PLANTED[name]
    assert text.count(old) == 1
    assert races(text.replace(old, new)) != []
