"""Kernels launched with programmatic stream serialization may start before the kernel ahead of them has completed: each
of them has to begin with grid_wait, before any access to memory, and reads what the kernel ahead wrote with plain loads."""
import pathlib
import re

import pytest

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2206_09878_gb300" / "csrc"
# launched with <<<>>> only: self-tests, rate probes, and the twiddles ahead of an ordinary launch
ORDINARY = {"k_tile_wait_probe", "k_df64_convert", "k_twiddles", "k_rate"}


def _kernels():
    for path in sorted(CSRC.glob("*.cu")):
        text = path.read_text()
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\([^;{]*\{\s*([^\n]*)", text):
            yield path.name, m.group(1), m.group(2)


def test_every_kernel_is_seen():
    names = [k for _, k, _ in _kernels()]
    declared = sum(len(re.findall(r"__global__", p.read_text())) for p in CSRC.glob("*.cu"))
    assert len(names) == declared and ORDINARY <= set(names)


@pytest.mark.parametrize("file,kernel,first", list(_kernels()), ids=lambda v: v if str(v).startswith("k_") else "")
def test_kernel_waits_first(file, kernel, first):
    if kernel in ORDINARY:
        assert first != "grid_wait();"
    else:
        assert first == "grid_wait();", (file, kernel)


def test_ordinary_kernels_are_launched_in_stream_order():
    text = "".join(p.read_text() for p in CSRC.glob("*.cu"))
    for k in ORDINARY:
        assert not re.search(r"(LMVD_LAUNCH\([^;]*|launch_next\()\b%s\b" % k, text), k


def test_exponents_written_by_the_pass_ahead_use_plain_loads():
    assert not re.search(r"__ldg\(\s*(ej|te)\b", (CSRC / "fft.cu").read_text())


def test_twiddles_of_an_overlapping_launch_use_plain_loads():
    """The allocation-free transform's z-pass overlaps the kernel that writes its twiddles only in the instantiation
    that reads them with plain loads (6 elements a thread)."""
    text = (CSRC / "fft.cu").read_text()
    assert len(re.findall(r"__ldg\(", text)) == 1 and "if constexpr (EPT == 12 && (S > 1 || SIGN > 0)) return __ldg(p);" in text
    entry = text[text.index("lmvd_inverse_transform_noalloc(int nx"):]
    assert re.findall(r"launch_next\((k_fft_z_inv<[^>]*>)", entry) == ["k_fft_z_inv<cd, 6, 4>"]
