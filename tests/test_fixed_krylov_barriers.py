"""The fixed-point Krylov kernel's magnitudes (the or and the largest of what every warp writes) are
cleared by one warp and gathered by all of them with atomics, so a barrier of the whole CTA lies
between the two: between every clearing in the kernel's step loop and the next phase that gathers."""
import os
import re

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1210_1531_gb300", "csrc",
                      "krylov_fixed.cu")
CLEAR = re.compile(r"st\.(bits|top)\[\d\]\[threadIdx\.x\] = [^;]*\b0;")


def source():
    with open(SOURCE) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def gathering_phases(text):
    """The device functions that end in the atomics."""
    return {re.findall(r"__forceinline__ void (fx_\w+)\(", text[:m.start()])[-1]
            for m in re.finditer(r"fx_(?:or|max)<NC>\(m", text)}


def unconditional(text):
    """The text without the blocks of its if statements."""
    while True:
        shorter = re.sub(r"\bif \((?:[^()]|\([^()]*\))*\) \{[^{}]*\}", "", text)
        if shorter == text:
            return text
        text = shorter


def test_a_barrier_follows_every_clearing():
    text = source()
    phases = gathering_phases(text)
    assert {"fx_update", "fx_products"} <= phases
    gather = re.compile(r"\b(%s)<" % "|".join(sorted(phases, key=len, reverse=True)))
    kernel = text[text.index(") k_krylov_fixed("):]
    kernel = kernel[:kernel.index("\nnamespace {")]
    assert phases == {m.group(1) for m in gather.finditer(kernel)}      # every one is called in the loop
    clears = [m.end() for m in CLEAR.finditer(kernel)]
    assert len(clears) >= 4
    for at in clears:
        following = gather.search(kernel, at)
        if following:
            assert "__syncthreads();" in unconditional(kernel[at:following.start()]), kernel[at - 80:following.end()]
