"""The MMA role of the CTA-pair attention kernel, compiled for the host as it stands in the source and run against a model of the other
roles with the rules of mbarrier (pair_mma_model.cpp): whatever the lengths of the units and the times at which they are published, no
QK^T or P V goes out before its operands are there."""
import pathlib
import subprocess

TESTS = pathlib.Path(__file__).resolve().parent
SOURCE = TESTS.parent / "paper_2409_12490_b200" / "csrc" / "attention_pair_sm100.cu"


def _between(text, first, end):
    at = text.index(first)
    return text[at:text.index(end, at)]


def test_no_product_is_issued_before_its_operands(tmp_path):
    text = SOURCE.read_text()
    role = tmp_path / "role.inc"
    role.write_text(_between(text, "constexpr int kThreads", "static_assert(sizeof(Bars)")
                    + _between(text, "template <bool kF16, int NS>\n__device__ __forceinline__ void mma_role(", "// -----"))
    exe = tmp_path / "model"
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", f'-DROLE_FILE="{role}"', "-o", str(exe), str(TESTS / "pair_mma_model.cpp")], check=True)
    out = subprocess.run([str(exe), "3000"], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr


def test_a_row_and_its_tag_are_exchanged_as_one_scalar():
    """PTX guarantees that a scalar access is seen whole; a vector access is one access per part."""
    text = SOURCE.read_text()
    for name, access in (("void row_put(", "st.volatile.shared.b64 "), ("uint2 row_load(", "ld.volatile.shared.b64 ")):
        body = _between(text, name, "\n}\n")
        assert body.count(access) == 1 and ".v2" not in body and body.count("asm volatile") == 1
