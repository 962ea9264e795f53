"""The bounds-checked build checks every access to the node bits and to the row
runs: in the sources, both arrays are subscripted, or their addresses handed
on, only behind in_bounds; and the words that a step addresses, restated, stay
inside the arrays' allocation (so that the checks skip nothing)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2308_16597_gb300", "csrc")


def code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//.*", "", f.read())


def test_node_bits_are_reached_through_checked_helpers_only():
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh")) or name == "lbm_api.cu":  # (the host's copies and clears)
            continue
        text = code(name)
        lines = [ln.strip() for ln in text.splitlines() if re.search(r"\bD\.bits\b", ln)]
        if name != "lbm_internal.cuh":
            assert lines == [], (name, lines)
        else:
            assert lines and all("bits_ok(" in ln or prev_checked(text, ln) for ln in lines), lines


def prev_checked(text, line):
    at = text.index(line)
    return "bits_ok(" in text[text.rfind("{", 0, at):at]


def test_row_runs_are_read_and_written_behind_a_check():
    text = code("k_particles.cu")
    uses = [ln.strip() for ln in text.splitlines() if re.search(r"\bD\.runs\b", ln)]
    # the checked read, and the raster's pointer whose one store is checked
    assert len(uses) == 2 and "in_bounds(" in uses[0], uses
    assert re.search(r"in_bounds\(D, \(long long\)p \* D\.zone_max \+ b0 \+ lane, \(long long\)D\.np \* D\.zone_max\)\)"
                     r"\s+runs\[b0 \+ lane\] =", text)
    assert len(re.findall(r"(?<!D\.)\bruns\[", text)) == 1


def test_bit_words_of_a_step_stay_inside_the_array():
    """Rows of bpitch = pitch / 32 words rounded up to 8, of both parities
    interleaved: every word that the window of a zone anywhere in the lattice,
    its clear and its raster touch, and every tile's copy, lies in
    [0, 2 bpitch ny)."""
    for nx in list(range(4, 300, 9)) + [512, 1023, 4000]:
        pitch = (nx + 31) // 32 * 32
        bpitch = (pitch // 32 + 7) // 8 * 8
        for ny in (4, 9):
            words = 2 * bpitch * ny
            for y in (0, ny - 1):
                for x in (0, nx - 1, pitch - 1):
                    w = 2 * (y * bpitch + x // 32)
                    assert 0 <= w and w + 1 < words
                for n in (5, 23, 60):  # clear and raster: columns clipped to the lattice
                    for x0 in range(-n, nx, max(1, nx // 7)):
                        w0, w1 = max(x0, 0) >> 5, min(x0 + n - 1, nx - 1) >> 5
                        for w in range(w0, w1 + 1):
                            assert 0 <= 2 * (y * bpitch + w) + 1 < words
                for xs in range(0, pitch, 256):  # a staged tile's copy of 64 bytes
                    w = 2 * (y * bpitch + xs // 32)
                    assert w % 4 == 0 and w + 16 <= words
