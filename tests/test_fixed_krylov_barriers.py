"""The fixed-point Krylov kernel's magnitudes (the or and the largest of what every warp writes) are
cleared by one warp and gathered by all of them with atomics, so a barrier of the whole CTA lies
between the two: between every clearing in the kernel's step loop and the next phase that gathers."""
import os
import re

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1210_1531_gb300", "csrc",
                      "krylov_fixed.cu")
CLEAR = re.compile(r"st\.(bits|top)\[\d\]\[threadIdx\.x\] = [^;]*\b0;")
GATHER = re.compile(r"\b(fx_update|fx_products|fx_products_lead|fx_products_dense)<")


def unconditional(text):
    """The text without the blocks of its if statements."""
    while True:
        shorter = re.sub(r"\bif \((?:[^()]|\([^()]*\))*\) \{[^{}]*\}", "", text)
        if shorter == text:
            return text
        text = shorter


def test_a_barrier_follows_every_clearing():
    with open(SOURCE) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    kernel = text[text.index(") k_krylov_fixed("):]
    kernel = kernel[:kernel.index("\nnamespace {")]
    clears = [m.end() for m in CLEAR.finditer(kernel)]
    assert len(clears) >= 4
    for at in clears:
        following = GATHER.search(kernel, at)
        end = following.start() if following else len(kernel)
        if following:
            assert "__syncthreads();" in unconditional(kernel[at:end]), kernel[at - 80:end + 20]


def test_the_gathers_are_where_the_loop_calls_them():
    """The phases the rule above looks for are the ones that end in the atomics."""
    with open(SOURCE) as f:
        text = f.read()
    names = set()
    for m in re.finditer(r"fx_(?:or|max)<NC>\(m", text):
        names.add(re.findall(r"__forceinline__ void (fx_\w+)\(", text[:m.start()])[-1])
    assert names == {"fx_products", "fx_products_dense", "fx_products_lead", "fx_update"}
