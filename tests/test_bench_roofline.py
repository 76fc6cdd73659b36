"""The ray pass's roofline counts rays that the benchmark run itself has counted,
for every workload: no share of evaluated rays is typed in."""
import ast
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_the_counted_rays_are_the_landed_ones():
    tree = ast.parse(open(os.path.join(ROOT, "bench.py")).read())
    shares = [ast.unparse(n.value) for n in ast.walk(tree) if isinstance(n, ast.Assign)
              and any(isinstance(t, ast.Name) and t.id == "share" for t in n.targets)]
    assert len(shares) == 2 and set(shares) == {"landed / info.n_rays"}, shares
