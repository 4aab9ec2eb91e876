"""An object or library is kept only while it is what its inputs make: a changed source, a missing file
or a build that was cut short is made again."""
from paper_2407_06409_gb300 import build


def test_targets_are_made_again_when_their_inputs_change(tmp_path):
    src, out = tmp_path / "a.cu", tmp_path / "a.o"
    cmd = [build._nvcc(), "-c", str(src), "-o", str(out)]
    src.write_text("int a;\n")
    first = build._digest(cmd, [str(src)])
    assert not build._up_to_date(str(out), first)          # nothing made yet
    out.write_text("object")
    build._made(str(out), first)
    assert build._up_to_date(str(out), first)
    assert build._digest([*cmd, "-G"], [str(src)]) != first
    src.write_text("int b;\n")
    second = build._digest(cmd, [str(src)])
    assert second != first and not build._up_to_date(str(out), second)
    assert not build._up_to_date(str(out), first)          # cut short after this: no digest is left
    build._made(str(out), first)
    out.unlink()
    assert not build._up_to_date(str(out), first)
