"""Runs a piece of Python against the emulated library: FACO_EMU=<library>
python run.py < code.  Prints what the code prints; ends with status 1 when
watched shared memory was reported."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
sys.path.insert(0, ROOT)

from paper_2203_02228_gb300 import build, load  # noqa: E402

build.LIB = os.environ["FACO_EMU"]
exec(compile(sys.stdin.read(), "<emulated>", "exec"))
sys.exit(1 if load().emu_take_reports() else 0)
