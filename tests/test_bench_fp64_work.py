"""The benchmark's FP64 operation counts against the ones stated at the kernel
(csrc/ddfd_step64.cu: 9 instructions a component of a plain node, 39 (36) for the Gauss-law
term), written out term by term for one node of each kind."""
import os

import bench

SRC = os.path.join(bench.ROOT, "paper_2508_07780_gb300", "csrc", "ddfd_step64.cu")


def per_node(*terms):
    """terms: (count, flops each); an operation is one instruction."""
    return sum(c for c, _ in terms), sum(c * f for c, f in terms)


def test_counts_follow_the_kernel():
    add, fma = 1, 2
    plain = per_node((3 * 5, add), (3, fma), (3, add), (3, fma), (3, add))
    fem = per_node((3, 1), (1, 1))                                        # A dv as a product, C = q2 r2
    diff, div, edge = (3, add), (6 * 2, add), (2 * 3 + 2 * 2 + 5 + 3, add)
    gauss_f = per_node((3, 1), diff, div, edge, (3, fma))
    gauss_a = per_node(diff, div, edge, (3, fma))
    grad = per_node((3 * 3, add), (3 * 2, fma), (1 + 3, 1), (2, add))
    assert (plain[0], gauss_f[0], gauss_a[0]) == (27, 39, 36)
    text = " ".join(open(SRC).read().split())
    assert "9 instructions a component" in text and "39 instructions a node (36 in // the adjoint)" in text
    for n, f in ((161, 121), (41, 21), (13, 5)):
        nodes, rows, free = n ** 3, (f - 2) ** 3, (f - 4) ** 3
        fwd, adj = bench.fp64_work(n, f)
        for q in range(2):
            assert fwd[q] == plain[q] * nodes + (fem[q] + gauss_f[q]) * rows
            assert adj[q] == plain[q] * nodes + fem[q] * rows + (gauss_a[q] + grad[q]) * free
