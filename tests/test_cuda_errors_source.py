"""The counting entry points name the CUDA error behind every TG_ECUDA: their source
(csrc/tg_count.cu) takes CUDA calls through TG_TRY_CUDA, which records the error for
tg_last_cuda_error, and never makes the status by itself.  Runs on the CPU."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1901_10026_gb300", "csrc")


def test_the_macro_records_the_error():
    text = open(os.path.join(CSRC, "tg_internal.cuh")).read()
    macro = text[text.index("#define TG_TRY_CUDA"):text.index("#define TG_TRY(call)")]
    assert "tg_note_cuda_error(_e)" in macro and "return TG_ECUDA" in macro


def test_counts_make_no_cuda_status_of_their_own():
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "tg_count.cu")).read())
    assert "TG_ECUDA" not in text
