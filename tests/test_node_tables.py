"""Host tables of the plan (host.cu: node_tables), printed by a small program linked with the library's host
object: the nodes are exactly symmetric about 0, as the kernels' mirror images of node pairs take
them to be, and accurate in the tails, against phi_i = pi i/(N+1) evaluated in extended precision."""
import numpy as np
import pytest

from _host_program import host_program

PROGRAM = """
int main(int argc, char **argv)
{
    for (int a = 1; a + 2 < argc; a += 3) {
        pgbh::NodeTables t = pgbh::node_tables(atoi(argv[a]), atof(argv[a + 1]), atoi(argv[a + 2]));
        for (size_t i = 0; i < t.v.size(); ++i) printf("%a %a %a ", t.v[i], t.scale_a[i], t.inv_mu2[i]);
        printf("\\n");
    }
}
"""


@pytest.fixture(scope="module")
def tables(tmp_path_factory):
    run = host_program(tmp_path_factory.mktemp("tables"), PROGRAM)
    return lambda args: [np.array([float.fromhex(x) for x in line.split()]).reshape(-1, 3).T for line in run(args)]


def test_nodes_are_exactly_symmetric_and_accurate(tables):
    cases = [(N, S, r) for N in (2, 3, 16, 41, 64, 121, 512) for S in (2.0, 3.25) for r in (0, 1)]
    for (N, S, r), (v, sa, im) in zip(cases, tables([x for c in cases for x in c])):
        assert np.array_equal(v, -v[::-1]) and np.array_equal(sa, sa[::-1]) and np.array_equal(im, im[::-1]), (N, S, r)
        pi = np.longdouble("3.14159265358979323846264338327950288")
        phi = pi * np.arange(1, N + 1, dtype=np.longdouble) / (N + 1)
        want = S * np.log(np.tan(phi / 2)) if r == 0 else -S * np.cos(phi) / np.sin(phi)
        # a handful of roundings (pi, phi, two functions, a quotient), each 1.1e-16 of the value or of S
        assert float((np.abs(v - want) / np.maximum(np.abs(want), S)).max()) < 2e-15, (N, S, r)
