"""Scratch that a streamed call sets aside before it goes through FP4 operands:
tests/host/stream_scratch_check.cu compares it with what every block's
comparison takes.  Host arithmetic only."""
import subprocess

from host import compile_against_library


def test_scratch_covers_every_block(tmp_path):
    exe = compile_against_library("stream_scratch_check.cu", str(tmp_path / "check"))
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout[-2000:]
    assert "bad 0" in r.stdout
