"""The FP64 instructions that mw_elementwise issues per operation (`bench.ELEMENTWISE_GPU_FP64`,
what its roofline counts), recounted as the nodes of the operation's expression graph that
the result's words need: two_sum is an addition for the sum and two for the error (its
operands are ordered on the integer units), fast_two_sum 3, two_prod a multiply and a
fused multiply-add, a division 1; products with a quotient word leave out its zero words.
CPU only."""
import pytest

import bench


class Graph:
    """Values are node numbers; args[v] the operands of v's instruction."""

    def __init__(self):
        self.args = []

    def node(self, *args):
        self.args.append(args)
        return len(self.args) - 1

    def leaf(self):
        return self.node()

    def count(self, outputs):
        """Instructions that the outputs depend on."""
        seen, todo = set(), list(outputs)
        while todo:
            v = todo.pop()
            if v is not None and v not in seen:
                seen.add(v)
                todo += self.args[v]
        return sum(1 for v in seen if self.args[v])

    def two_sum(self, a, b):
        s = self.node(a, b)
        return s, self.node(a, b, self.node(a, b, s))

    fast_two_sum = two_sum

    def two_prod(self, a, b):
        p = self.node(a, b)
        return p, self.node(a, b, p)

    def renorm(self, x, m):
        x, r = list(x), []
        for _ in range(m):
            if not x:
                r.append(None)                     # a zero word
                continue
            s, errs = x[-1], [None] * len(x)
            for i in range(len(x) - 2, -1, -1):
                s, errs[i + 1] = self.two_sum(x[i], s)
            r.append(s)
            x = errs[1:]
        return r

    def add(self, a, b):
        if len(a) == 2:
            s, e = self.two_sum(a[0], b[0])
            t, f = self.two_sum(a[1], b[1])
            s, e = self.fast_two_sum(s, self.node(e, t))
            return list(self.fast_two_sum(s, self.node(e, f)))
        return self.renorm([v for w in zip(a, b) for v in w], len(a))

    def mul(self, a, b):
        m = len(a)
        if m == 2:
            p, e = self.two_prod(a[0], b[0])
            cross = self.node(self.node(a[0], b[1]), self.node(a[1], b[0]))
            return list(self.fast_two_sum(p, self.node(e, cross)))
        t, lo = [], []
        for level in range(m):
            hi = [self.two_prod(a[i], b[level - i]) for i in range(level + 1)]
            t += [p for p, _ in hi] + lo
            lo = [e for _, e in hi]
        t += [self.node(a[i], b[m - i]) for i in range(1, m)]
        return self.renorm(t + lo, m)

    def mul_word(self, q, b):
        m = len(b)
        if m == 2:
            p, e = self.two_prod(q, b[0])
            return list(self.fast_two_sum(p, self.node(e, self.node(q, b[1]))))
        t, lo = [], []
        for w in b:
            p, e = self.two_prod(q, w)
            t += [p] + lo
            lo = [e]
        return self.renorm(t + lo, m)

    def div(self, a, b):
        m, rem, q = len(a), a, []
        for i in range(m + 1):
            q.append(self.node(rem[0], b[0]))
            if i < m:
                rem = self.add(rem, self.mul_word(q[i], b))
                if m > 2:
                    rem = self.renorm(rem, m)
        return self.renorm(q, m)


@pytest.mark.parametrize("op", ["add", "mul", "div"])
@pytest.mark.parametrize("m", [2, 4, 8])
def test_instructions_issued(m, op):
    g = Graph()
    a, b = [g.leaf() for _ in range(m)], [g.leaf() for _ in range(m)]
    assert g.count(getattr(g, op)(a, b)) == bench.ELEMENTWISE_GPU_FP64[m][op]
