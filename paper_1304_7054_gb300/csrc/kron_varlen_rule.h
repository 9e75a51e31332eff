// How a mixed-size launch spreads its tiles (plain arithmetic, also for the host tests).
#pragma once

namespace kron {

// Whether one CTA per tile is launched and running CTAs take over the rest, so that the
// tiles are worked off in the order of the list (else the resident CTAs walk it in fixed
// steps).  Code of many large classes wants that order; a class's is about 24 bytes times
// kind n^2 (units: their sum), and below about 17 KB the instruction cache holds all of it:
// there walked tiles are 3-5% faster (3-D n = 16 alone: 90 us walked, 86 taken in order;
// n = 6 alone: 68 and 70).  Lists of up to two tiles for each resident CTA are walked too,
// because the requests delay the first tiles (3-D n = 8..12, 2000 instances: 14.6 us taken
// over, 12.5 walked; 2-D n = 4..16, 20,000: 18.7 and 16.7; n = 2..16, 20,000: 19.4 and 18.5).
inline bool tiles_taken_over(int units, int tiles, int resident) { return units >= 700 && tiles > 2 * resident; }

}  // namespace kron
