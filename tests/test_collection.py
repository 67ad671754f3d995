"""CPU: every test function of this folder is collected, from its own file, also when the files are collected together."""
import ast
import pathlib
import subprocess
import sys

HERE = pathlib.Path(__file__).resolve().parent


def _defined():
    for path in sorted(HERE.glob("test_*.py")):
        for node in ast.parse(path.read_text()).body:
            if isinstance(node, ast.FunctionDef) and node.name.startswith("test_"):
                yield path.name, node.name


def test_every_test_function_is_collected():
    out = subprocess.run([sys.executable, "-m", "pytest", "--collect-only", "-q", "-p", "no:cacheprovider", str(HERE)],
                         capture_output=True, text=True, cwd=HERE.parent)
    assert out.returncode == 0, out.stdout[-2000:] + out.stderr[-2000:]
    collected = set()
    for line in out.stdout.splitlines():
        parts = line.strip().split("::")
        if len(parts) == 2:
            collected.add((pathlib.PurePath(parts[0]).name, parts[1].split("[")[0]))
    missing = sorted(set(_defined()) - collected)
    assert not missing, missing
    # (a test imported under its own name would run a second time there)
    assert not sorted(collected - set(_defined()))
