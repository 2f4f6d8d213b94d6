"""The shared words of the one-kernel charge solve, read off its source: one
thread of a block stores the scalars and decisions that all threads read, so a
word read by all may be stored again only past a barrier, and may be read only
past the barrier after its store. The kernel's statements are followed in the
order of execution (both sides of every branch, loops until nothing changes,
lambdas where they are called) in both precisions."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1802_07871_gb300", "csrc")
WORDS = ("s_stop", "s_fell", "s_shift", "s_abc", "s_tot")
EVENT = re.compile(r"\b(?P<word>" + "|".join(WORDS) + r")\b(?P<store>(?:\[[^\]]*\])?\s*=(?!=))?|(?P<call>\b\w+\s*(?:<[^<>;()]*>)?)\(")


def _close(t, i):
    """Index past the bracket that closes t[i]."""
    pairs, depth = {"{": "}", "(": ")", "[": "]"}, 0
    a, b = t[i], pairs[t[i]]
    for k in range(i, len(t)):
        depth += (t[k] == a) - (t[k] == b)
        if depth == 0:
            return k + 1
    raise ValueError("unbalanced source")


def _parse(t, lambdas):
    """Statements of t: ("text", s), ("if", cond, then, else), ("loop", head, body)."""
    out, i = [], 0

    def body(i):
        if t[i] == "{":
            e = _close(t, i)
            return _parse(t[i + 1:e - 1], lambdas), e
        e = i
        m = re.compile(r"(if|for|while)\b").match(t, i)
        if m:
            node, e = statement(i)
            return [node], e
        while t[e] != ";":
            e = _close(t, e) if t[e] in "({[" else e + 1
        return [("text", t[i:e])], e + 1

    def skip(i):
        while i < len(t) and t[i].isspace():
            i += 1
        return i

    def statement(i):
        m = re.compile(r"(if)\s*(?:constexpr\s*)?(?=\()|(for|while)\s*(?=\()").match(t, i)
        p = _close(t, m.end())
        head = t[m.end():p]
        then, e = body(skip(p))
        if m.group(2):
            return ("loop", head, then), e
        other, k = [], skip(e)
        if t.startswith("else", k):
            other, e = body(skip(k + 4))
        return ("if", head, then, other), e

    while (i := skip(i)) < len(t):
        m = re.compile(r"auto\s+(\w+)\s*=\s*\[&\]\s*(?=\()").match(t, i)
        if m:
            b = t.index("{", _close(t, m.end()))
            e = _close(t, b)
            lambdas[m.group(1)] = _parse(t[b + 1:e - 1], lambdas)
            i = e + 1
        elif m := re.compile(r"do\s*(?=\{)").match(t, i):   # (once)
            e = _close(t, m.end())
            out += _parse(t[m.end() + 1:e - 1], lambdas)
            i = t.index(";", e) + 1
        elif t[i] == "{":
            e = _close(t, i)
            out += _parse(t[i + 1:e - 1], lambdas)
            i = e
        elif re.compile(r"(if|for|while)\s*(constexpr\s*)?\(").match(t, i):
            node, i = statement(i)
            out.append(node)
        else:
            e = i
            while t[e] != ";":
                e = _close(t, e) if t[e] in "({[" else e + 1
            out.append(("text", t[i:e]))
            i = e + 1
    return out


class _Walk:
    """Follows the statements with the set of possible states: the words that
    all threads read, and those that were stored, since the last barrier."""

    def __init__(self, lambdas, size):
        self.lambdas, self.size = lambdas, size
        self.bad, self.barriers = set(), 0

    def barrier(self, states):
        self.barriers += 1
        return {(frozenset(), frozenset())}

    def store(self, states, word):
        if any(word in r for r, _ in states):
            self.bad.add(f"{word} stored with no barrier after a read")
        return {(r, s | {word}) for r, s in states}

    def read(self, states, word, boss):
        if boss:
            return states
        if any(word in s for _, s in states):
            self.bad.add(f"{word} read with no barrier after its store")
        return {(r | {word}, s) for r, s in states}

    def run(self, nodes, states, boss=False):
        for n in nodes:
            states = self.text(n[1], states, boss)
            if n[0] == "loop":
                while True:
                    more = states | self.run(n[2], states, boss)
                    more |= self.text(n[1], more, boss)
                    if more == states:
                        break
                    states = more
            elif n[0] == "if":
                cond = n[1][1:-1].strip()
                m = re.fullmatch(r"sizeof\(R\) == (\d)", cond)
                if cond == "boss":
                    states = self.run(n[2], states, True)
                elif m:
                    states = self.run(n[2] if int(m.group(1)) == self.size else n[3], states, boss)
                else:
                    states = self.run(n[2], states, boss) | self.run(n[3], states, boss)
        return states

    def text(self, s, states, boss):
        after, i = [], 0
        while m := EVENT.search(s, i):
            i = m.end()
            if m.group("word"):
                if m.group("store"):
                    after.append(m.group("word"))   # (after the reads of its right-hand side)
                else:
                    states = self.read(states, m.group("word"), boss)
                continue
            name = re.split(r"\W", m.group("call").strip())[0]
            e = _close(s, m.end() - 1)
            if name == "__syncthreads":
                states = self.barrier(states)
            elif name == "exchange":
                # stores the totals between two of its own barriers (its
                # arguments name s_tot only to pass it on)
                states = self.barrier(self.store(self.barrier(states), "s_tot"))
                i = e
            elif name in self.lambdas:
                states = self.text(s[m.end():e - 1], states, boss)
                states = self.run(self.lambdas[name], states, boss)
                i = e
        for word in after:
            states = self.store(states, word)
        return states


def _kernel(text):
    text = re.sub(r"//[^\n]*|^\s*#[^\n]*", "", text, flags=re.M)
    k = text.index("k_cg_solve(const SolveArgs")
    b = text.index("{", k)
    return text[b + 1:_close(text, b) - 1]


def _check(text, size):
    lambdas = {}
    nodes = _parse(_kernel(text), lambdas)
    assert {"test", "iterate", "exchange1", "exchange_y", "precond"} <= set(lambdas)
    walk = _Walk(lambdas, size)
    walk.run(nodes, {(frozenset(), frozenset())})
    assert walk.barriers > 10   # (the solve's loop was followed)
    return walk.bad


@pytest.mark.parametrize("size", [4, 8])
def test_words_are_stored_and_read_across_barriers(size):
    with open(os.path.join(CSRC, "cgsolve.cu")) as f:
        assert _check(f.read(), size) == set()


def test_the_check_sees_a_missing_barrier():
    src = '''k_cg_solve(const SolveArgs<R> A) {
      auto exchange1 = [&](double v) { return T.template exchange<1, false>(own, v, s_tot); };
      auto exchange_y = [&](double v) { return T.template exchange<2, true>(own, v, s_tot); };
      auto precond = [&](double r) { return r; };
      auto test = [&](double sr) { s_stop = sr < 1.0; };
      auto iterate = [&](double r) { for (int k = 0; k < n; ++k) { exchange_y(r); } return true; };
      for (int cycle = 0;; ++cycle) {
        if (!exchange1(q)) break;
        if (boss) test(s_tot[0]);
        __syncthreads();
        conv = s_stop;
        if (conv) break;
        %s
        if (boss) s_stop = 1;
        __syncthreads();
        iterate(q);
        iterate(s_stop);
      }
    }'''
    assert _check(src % "__syncthreads();", 8) == set()
    assert _check(src % "", 8) == {"s_stop stored with no barrier after a read"}
