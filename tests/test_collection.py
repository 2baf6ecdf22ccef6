"""Every test function that the files of this folder define is collected when
the folder is collected as a whole: a module that imports another's test to
reuse its body must not take it out of the run."""
import ast
import glob
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))


def test_every_test_function_is_collected():
    defined = set()
    for path in glob.glob(os.path.join(HERE, "test_*.py")):
        tree = ast.parse(open(path).read())
        defined |= {os.path.basename(path) + "::" + f.name for f in tree.body
                    if isinstance(f, ast.FunctionDef) and f.name.startswith("test")}
    r = subprocess.run([sys.executable, "-m", "pytest", HERE, "--collect-only", "-q", "-p", "no:cacheprovider"],
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    collected = {os.path.basename(line.split("[")[0].strip()) for line in r.stdout.splitlines() if "::" in line}
    assert len(defined) > 50 and not defined - collected, sorted(defined - collected)
