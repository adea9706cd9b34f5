"""When the autograd node is built again: it depends on torch's and Python's binary interfaces, not on its sources alone."""
import os


def test_a_node_for_another_torch_is_stale(tmp_path, monkeypatch):
    from paper_2510_27527_b200 import build

    lib = tmp_path / "_node.so"
    assert build._node_stale(str(lib), build.NODE_SOURCES)
    lib.write_bytes(b"..." + build.node_tag().encode() + b"\0...")
    assert not build._node_stale(str(lib), build.NODE_SOURCES)
    for tag in ("torch 9.0.0, cpython-312-x86_64-linux-gnu", build.node_tag()[:-1]):
        monkeypatch.setattr(build, "node_tag", lambda tag=tag: tag)
        assert build._node_stale(str(lib), build.NODE_SOURCES)
    monkeypatch.undo()
    os.utime(lib, (0, 0))  # older than its sources
    assert build._node_stale(str(lib), build.NODE_SOURCES)


def test_the_built_node_says_what_it_is_for():
    from paper_2510_27527_b200 import _node, build

    assert _node.built_for == build.node_tag()
