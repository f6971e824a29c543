"""What the build step compiles again, with a stand-in for the compiler that notes its calls."""
import os

import pytest

from paper_2510_11400_b200 import build


@pytest.fixture
def calls(tmp_path, monkeypatch):
    log = tmp_path / "calls"
    nvcc = tmp_path / "nvcc"
    nvcc.write_text(f'#!/bin/sh\necho "$@" >> {log}\ncase "$*" in *broken*) exit 1;; esac\n'
                    'while [ "$1" != -o ]; do shift; done\necho made > "$2"\n')
    nvcc.chmod(0o755)
    monkeypatch.setenv("PATH", f"{tmp_path}:{os.environ['PATH']}")
    sources = [tmp_path / "a.cu", tmp_path / "b.cu"]
    for s in sources:
        s.write_text("")
    monkeypatch.setattr(build, "SOURCES", [str(s) for s in sources])
    monkeypatch.setattr(build, "HEADERS", [])
    monkeypatch.setattr(build, "DEPS", [str(s) for s in sources])
    monkeypatch.setattr(build, "OBJDIR", str(tmp_path / "objects"))
    monkeypatch.setattr(build, "LIB", str(tmp_path / "lib.so"))

    def take():
        lines = log.read_text().splitlines() if log.exists() else []
        log.write_text("")
        return [" ".join(w for w in ln.split() if w.endswith((".cu", "-shared"))) for ln in lines]
    return take


def compiled(lines):
    return sorted(os.path.basename(ln) for ln in lines)


def test_only_what_is_out_of_date_is_compiled(calls):
    build.build()
    assert compiled(calls()) == ["-shared", "a.cu", "b.cu"]
    build.build()
    assert calls() == []
    later = os.path.getmtime(build.LIB) + 5
    os.utime(build.SOURCES[0], (later, later))
    build.build()
    assert compiled(calls()) == ["-shared", "a.cu"]


def test_objects_made_with_other_flags_are_not_used(calls, monkeypatch):
    build.build()
    calls()
    monkeypatch.setattr(build, "FLAGS", build.FLAGS + ["-G"])
    os.remove(build.LIB)
    build.build()
    assert compiled(calls()) == ["-shared", "a.cu", "b.cu"]


def test_a_failed_build_leaves_nothing_that_looks_complete(calls, tmp_path, monkeypatch):
    bad = tmp_path / "broken.cu"
    bad.write_text("")
    monkeypatch.setattr(build, "SOURCES", build.SOURCES + [str(bad)])
    with pytest.raises(RuntimeError):
        build.build()
    assert not os.path.exists(build.LIB) and not [f for f in os.listdir(build.OBJDIR) if "broken" in f or "tmp" in f]


def test_the_flags_file_is_a_dependency_and_the_command_line_builds_anew():
    assert os.path.abspath(build.__file__) in build.DEPS
    source = open(build.__file__).read()
    assert "build(force=True" in source[source.index("__main__"):]
