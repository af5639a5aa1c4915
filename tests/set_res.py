"""Generated REs over two to four letters whose runs tend to stay apart: bounded repeats of the whole
alphabet, words, and unions of unequal lengths under stars."""
import random


def generated(seed, count):
    """(RE, alphabet) pairs from the seed alone."""
    rng = random.Random(seed)
    out = []
    for _ in range(count):
        al = rng.choice(["ab", "abc", "ACGT"])
        cls = "[" + al + "]"

        def word():
            return "".join(rng.choice(al) for _ in range(rng.randint(1, 4)))

        def unit():
            r, n = rng.random(), rng.randint(2, 6)
            if r < 0.35:
                return cls + "{%d}" % n
            if r < 0.5:
                return cls + "{%d,%d}" % (n, n + 1)
            return word() if r < 0.8 else word() + cls + "{%d}" % rng.randint(1, 3)

        def union():
            return "(" + "|".join("".join(unit() for _ in range(rng.randint(1, 3))) for _ in range(rng.randint(1, 3))) + ")"

        src = "(" + union() + "*" + word() + ")*" if rng.random() < 0.5 else union() + "*"
        if rng.random() < 0.5:
            src += rng.choice([cls + "*", union() + "*", word()])
        out.append((src, al.encode()))
    return out
