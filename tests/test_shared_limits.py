"""The shared-memory limit of the node-list kernel (csrc/op.cu) where two host
threads' launches meet: the other thread's call runs between the setting of the
limit and the launch, with planes on both sides of the default limit and of what
asks for more."""

import os

import fake_device


def test_node_lists_of_two_threads(tmp_path):
    from paper_1107_5719_gb300 import build as B
    B.build()
    folder = str(tmp_path)
    objs = [os.path.join(B.BUILD, "op.o"),
            fake_device.compile_cpp("list_limit.cpp", os.path.join(folder, "list_limit.o"))]
    exe = os.path.join(folder, "list_limit")
    fake_device.sh("g++", "-o", exe, *objs, fake_device.stubs(objs, folder))
    rows = [list(map(int, line.split())) for line in fake_device.sh(exe).splitlines()]
    assert len(rows) == 24
    assert any(launches == 2 for _, _, launches, _ in rows)
    assert not [r for r in rows if r[3]]
